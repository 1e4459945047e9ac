// tqp_filter: predicate evaluation + stream compaction + fused projection-sum.
//
// Paper Section 3.1 (Listing 1: comparison mask then masked_select; the
// selection-vector variant uses nonzero + index_select) and Section 5.1
// (expressions).  Two kernels, no host synchronisation and no inter-CTA
// waiting on the streaming path:
//   k_filter   the staged scan: the producer warp stages the predicate
//              columns in shared memory with bulk asynchronous copies; consumer
//              warps evaluate the conjunction lane-per-row, take one warp
//              ballot per 32 rows and store it (a 1-bit-per-row selection
//              mask, 1/128 of a 16-byte row), count with popc into per-block
//              totals, and evaluate the sum expression for passing rows only
//              (columns that are not staged are read lazily);
//   k_compact  expands the mask (written moments before, so read from L2)
//              into ascending int32 row ids: each block takes the total of all
//              earlier blocks as its offset, then scans its own words with
//              warp ballots/shuffles and writes ids with coalesced stores.
// Count and sum are reduced per warp and added once per warp to scratch; the
// last warp to finish publishes them.
//
// An earlier single-kernel form that chained tiles with a decoupled look-back
// (per tile, then per chunk) was measured slower on GB300: per-tile look-back
// advances the published-prefix frontier only ~32 tiles per L2 round trip, and
// a per-chunk look-back leaves the expansion as a serial tail.  The offsets
// here come straight from counts that are complete when k_compact starts.
#include <mutex>

#include <cstdio>

#include "host.h"
#include "bodies.cuh"
#include "filterdirect.cuh"

namespace tqp {



// Scratch layout (bytes): ticket + acc[3], block totals, then the mask.
struct FilterScratch {
    size_t tot_off, mask_off, bytes;
    long long nblocks;
};

static FilterScratch filter_scratch_layout(long long n, long long mask_rows, bool ids) {
    FilterScratch s;
    s.nblocks = ids ? (n + kCompactRows - 1) / kCompactRows : 0;
    s.tot_off = 4 * sizeof(unsigned long long);
    s.mask_off = (s.tot_off + s.nblocks * sizeof(uint32_t) + 255) / 256 * 256;
    s.bytes = s.mask_off + (ids ? static_cast<size_t>(mask_rows / kWarp) * sizeof(uint32_t) : 0);
    return s;
}


__global__ void __launch_bounds__(kEngineThreads, 2) k_filter(const __grid_constant__ FilterArgs P) {
    extern __shared__ __align__(128) unsigned char smem[];
    const FilterArgs& A = stage_args(P, smem + kHeaderBytes);
    FilterBody body(A, smem + kHeaderBytes + args_bytes<FilterArgs>());
    run_engine(A.G, A.ctl, body, smem, args_bytes<FilterArgs>());
}

// Variant 1, the built-in form but for plain_loads_win: plain vector loads
// (filterdirect.cuh). The staged scan (variant 0) keeps what falls outside its
// shapes -- no condition, more than four, more than two on 64-bit columns, three
// on 32-bit or two on 8-bit ones, sums that are not products of two affine
// factors -- and launch shapes set by the caller.
__global__ void __launch_bounds__(kFdThreads, kFdMinBlocks) k_filter_direct(const __grid_constant__ FilterDirectArgs A) {
    filter_direct_block(A, blockIdx.x, gridDim.x);
}

// The form of a filter, -1 for the built-in choice: the tuner's for calls of
// tqp_filter; in a plan or a shared scan the tuned variant is that operator's.
static int filter_variant(const tqp_ctx* ctx) {
    if (ctx->force_variant >= 0) return ctx->force_variant;
    return strncmp(ctx->cur_key, "filter ", 7) == 0 ? tuned_variant(ctx, -1) : -1;
}

// Built in: the plain loads, but without a sum the staged scan for a few mixes
// whose steps of plain loads have too few bytes in flight for what they wait, and
// which the staged scan streams faster. Plain / staged time, counts only (with row
// ids), 5% of the rows passing:
//   rows                       4.5M       8M          24M         60M         140M
//   two int64               0.92 (.94) 1.06 (1.05) 1.11 (1.15) 1.10 (1.09) 1.01 (1.04)
//   with an uint8           0.96 (1.0) 1.17 (1.19) 1.18 (1.14) 1.09 (1.09) 1.02 (1.04)
//   int64, two int32        0.96 (.94) 1.12 (1.10) 1.12 (1.12) 1.08 (1.10) 1.04 (1.07)
//   int64, int32, uint8     0.89 (.94) 1.06 (1.10) 1.06 (1.05) 1.00 (1.02) 0.96 (1.00)
//   with another int32      0.93 (.94) 1.11 (1.07) 1.08 (1.06) 1.03 (1.03) 0.98 (1.00)
//   with another uint8      0.89 (.94) 1.08 (1.07) 1.04 (1.01) 0.96 (1.00) 0.92 (0.97)
//   int64, int32            0.87 (.90) 0.91 (0.95) 1.00 (1.00) 1.04 (0.97) 0.95 (0.93)
// and 1.05 for the last one's counts at 40M and 50M. Every other mix takes 0.64 to
// 1.04 of the staged time from 2^23 rows on (int64 and three int32 0.72 to 0.91, two
// int64 and an int32 0.78 to 1.02). With a sum the plain loads read its columns only
// where rows pass: int64 and two int32 at 24M rows take 1.14 of the staged time with
// 5% of the rows passing, 0.97 with 50%, 0.45 with 95% of each condition.
static bool plain_loads_win(const FilterDirectArgs& D, bool ids) {
    const long long n = D.n;
    if (D.has_sum || n < (5LL << 20)) return true;
    if (D.nwide == 2 && D.nword == 0) {
        if (D.nbyte == 0) return n < (1LL << 23) || (!ids && n >= (1LL << 27));
        return D.nbyte != 1;
    }
    if (D.nwide != 1) return true;
    if (D.nword == 2 && D.nbyte == 0) return false;
    if (D.nword >= 1 && D.nbyte == 1) return n >= (1LL << 26);
    if (D.nword == 1 && D.nbyte == 2) return n >= (1LL << 25);
    if (D.nword == 1 && D.nbyte == 0) return ids || n < (1LL << 25) || n >= (1LL << 26);
    return true;
}

__global__ void __launch_bounds__(kCompactThreads) k_compact(const uint32_t* __restrict__ mask,
                                                             const uint32_t* __restrict__ block_tot, long long n,
                                                             int32_t* __restrict__ row_ids, long long capacity) {
    compact_block(mask, block_tot, n, row_ids, capacity, blockIdx.x);
}

bool lower_filter_direct(const tqp_table* t, const FilterArgs& F, FilterDirectArgs* A) {
    if (F.ncond < 1 || F.ncond > kFdConds) return false;
    ScanGeom G;
    memset(&G, 0, sizeof(G));
    G.n = t->num_rows;
    G.ncols = t->num_cols;
    for (int c = 0; c < t->num_cols; ++c) {
        G.col[c].type = t->cols[c].type;
        G.col[c].slot = 0;
        G.col[c].soff = c;
    }
    auto ptr = [&](int c) { return static_cast<const unsigned char*>(t->cols[c].data); };
    auto type = [&](int c) {
        const bool a32 = reinterpret_cast<uintptr_t>(t->cols[c].data) % 32 == 0;
        return t->cols[c].type == TQP_I64 && a32 ? kFdI64A32 : t->cols[c].type;
    };
    CondFast cf[TQP_MAX_PREDS];
    int32_t fast = 0;
    lower_fast(F.cond, F.ncond, G, cf, &fast);
    if (!fast) return false;
    memset(A, 0, sizeof(*A));
    A->n = t->num_rows;
    A->steps = kFdSteps;
    int k = 0;
    for (const int32_t want : {TQP_I64, TQP_I32, TQP_U8}) {
        const int first = k;
        for (int q = 0; q < F.ncond; ++q) {
            if (cf[q].type != want) continue;
            const uint64_t full = want == TQP_I64 ? ~0ULL : 0xFFFFFFFFULL;
            uint64_t lo = static_cast<uint64_t>(cf[q].lo), span = cf[q].span & full;
            if (cf[q].negate) {
                if (span == full) return false;  // never true
                lo += span + 1;
                span = full - span - 1;
            }
            A->cond[k++] = FdCond{ptr(cf[q].soff), type(cf[q].soff) == kFdI64A32, 0, lo, span};
        }
        const int m = k - first;
        if (want == TQP_I64) A->nwide = m;
        else if (want == TQP_I32) A->nword = m;
        else A->nbyte = m;
    }
    if (k != F.ncond || A->nwide > kFdWide || A->nword > kFdWord || A->nbyte > kFdByte) return false;
    A->has_sum = F.has_sum;
    if (F.has_sum) {
        ProdForm pf;
        if (!lower_prod(F.sum, G, &pf)) return false;
        for (int k = 0; k < 2; ++k) {
            const bool col = pf.kind[k] != kFacConst;
            A->f[k] = PjFactor{col ? ptr(pf.soff[k]) : nullptr, col ? type(pf.soff[k]) : 0, pf.kind[k], pf.a[k], pf.b[k]};
        }
    }
    return true;
}

// Lower a filter call's conditions and sum, and check its columns; *staged and
// *staged_bytes: the columns a staged scan copies, and their bytes per row.
static tqp_status lower_filter(const tqp_table* t, const tqp_pred* preds, int32_t npreds, const tqp_expr* sum_expr,
                               FilterArgs* A, std::vector<int>* staged_cols, int* staged_bytes) {
    memset(A, 0, sizeof(*A));
    int ncond = 0;
    TQP_TRY(lower_preds(t, preds, npreds, A->cond, &ncond));
    A->ncond = ncond;
    std::vector<int>& staged = *staged_cols;
    for (int i = 0; i < ncond; ++i) staged.push_back(A->cond[i].col);
    if (sum_expr) {
        TQP_TRY(lower_expr(sum_expr, t->num_cols, &A->sum));
        A->has_sum = 1;
        if (ncond == 0) expr_cols(A->sum, staged);  // every row passes: stage the summed columns
    }
    std::vector<int> u = staged;
    std::sort(u.begin(), u.end());
    u.erase(std::unique(u.begin(), u.end()), u.end());
    TQP_TRY(check_device_cols(t, u, "tqp_filter"));
    if (A->has_sum) {  // the rest are read in place at passing rows only
        std::vector<int> lazy;
        expr_cols(A->sum, lazy);
        TQP_TRY(check_numeric_cols(t, lazy, "tqp_filter sum_expr"));
        TQP_TRY(check_visible_cols(t, lazy, "tqp_filter"));
    }
    int bpr = 0;
    for (int c : u) bpr += t->cols[c].type == TQP_I64 ? 8 : (t->cols[c].type == TQP_I32 ? 4 : 1);
    *staged_bytes = bpr;
    return TQP_OK;
}

// The launch shape of a lowered filter as a staged scan.
static tqp_status shape_filter(const tqp_ctx* ctx, const tqp_table* t, const std::vector<int>& staged, int bpr, bool ids,
                               const tqp_tuning* force, FilterArgs* A, size_t* smem, int* grid, FilterScratch* lay) {
    const tqp_tuning tu = force ? *force : default_tuning(ctx, bpr, FilterBody::kSmemBytes + args_bytes<FilterArgs>());
    TQP_TRY(make_geom(ctx, t, staged, tu, FilterBody::kSmemBytes + args_bytes<FilterArgs>(), &A->G, smem));
    lower_fast(A->cond, A->ncond, A->G, A->cf, &A->fast);
    static SmemFlags attr_done;
    TQP_TRY(allow_smem(ctx, reinterpret_cast<const void*>(k_filter), attr_done));
    const int g = engine_grid(ctx, reinterpret_cast<const void*>(k_filter), *smem, A->G.ntiles, tu.ctas_per_sm);
    A->ctl.chunk_tiles = (A->G.ntiles + g - 1) / g;
    A->ctl.nchunks = (A->G.ntiles + A->ctl.chunk_tiles - 1) / A->ctl.chunk_tiles;
    *grid = static_cast<int>(A->ctl.nchunks);
    *lay = filter_scratch_layout(A->G.n, A->G.ntiles * A->G.T, ids);
    return TQP_OK;
}

// Launch with caller-provided scratch of at least lay.bytes (cleared here).
static tqp_status launch_filter_with(FilterArgs& A, int grid, size_t smem, const FilterScratch& lay,
                                     void* scratch, int* d_err, long long wait_cap, int32_t* d_row_ids,
                                     int64_t capacity, int64_t* d_count, int64_t* d_sum, cudaStream_t stream,
                                     FilterDirectArgs* direct = nullptr, int direct_grid = 0) {
    unsigned char* sc = static_cast<unsigned char*>(scratch);
    TQP_CUDA(cudaMemsetAsync(sc, 0, lay.mask_off, stream));
    A.ctl.ticket = reinterpret_cast<unsigned long long*>(sc);
    A.ctl.err = d_err;
    A.ctl.wait_cap = wait_cap;
    A.acc = reinterpret_cast<unsigned long long*>(sc) + 1;
    A.block_tot = reinterpret_cast<uint32_t*>(sc + lay.tot_off);
    A.mask = d_row_ids ? reinterpret_cast<uint32_t*>(sc + lay.mask_off) : nullptr;
    A.capacity = capacity;
    A.d_count = d_count;
    A.d_sum = d_sum;
    if (direct) {
        direct->mask = A.mask;
        direct->block_tot = A.block_tot;
        direct->acc = A.acc;
        direct->d_count = d_count;
        direct->d_sum = d_sum;
        direct->capacity = capacity;
        direct->err = d_err;
        k_filter_direct<<<direct_grid, kFdThreads, 0, stream>>>(*direct);
    } else {
        k_filter<<<grid, kEngineThreads, smem, stream>>>(A);
    }
    TQP_CUDA(cudaGetLastError());
    if (d_row_ids) {
        k_compact<<<static_cast<unsigned>(lay.nblocks), kCompactThreads, 0, stream>>>(A.mask, A.block_tot, A.G.n,
                                                                                       d_row_ids, capacity);
        TQP_CUDA(cudaGetLastError());
    }
    return TQP_OK;
}

tqp_status launch_filter(tqp_ctx* ctx, const tqp_table* t, const tqp_pred* preds, int32_t npreds,
                         const tqp_expr* sum_expr, int64_t* d_sum, int32_t* d_row_ids, int64_t capacity,
                         int64_t* d_count, cudaStream_t stream, const tqp_tuning* force) {
    // IN / LIKE / NOT LIKE: one pre-pass writes a pass column that the scan then filters on
    StrLowered SL;
    TQP_TRY(str_prepass(ctx, t, preds, npreds, stream, &SL));
    if (SL.active) {
        t = &SL.t;
        preds = SL.preds;
        npreds = SL.npreds;
    }
    FilterArgs A;
    size_t smem = 0;
    int grid = 0;
    FilterScratch lay;
    std::vector<int> staged;
    int bpr = 0;
    TQP_TRY(lower_filter(t, preds, npreds, sum_expr, &A, &staged, &bpr));
    const long long n = t->num_rows;
    if (n == 0) {
        TQP_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int64_t), stream));
        if (d_sum) TQP_CUDA(cudaMemsetAsync(d_sum, 0, sizeof(int64_t), stream));
        return TQP_OK;
    }
    const bool ids = d_row_ids != nullptr;
    FilterDirectArgs D;
    const int variant = filter_variant(ctx);
    const bool plain = !force && !user_shape(ctx) && variant != 0 && lower_filter_direct(t, A, &D);
    auto run_plain = [&]() -> tqp_status {
        lay = filter_scratch_layout(n, (n + kFdStep - 1) / kFdStep * kFdStep, ids);
        void* scratch = arena_alloc(ctx, lay.bytes);
        if (!scratch) return arena_oom(ctx, lay.bytes);
        const long long step = kFdStep * (kFdThreads / kWarp), most = 1LL * kFdMinBlocks * ctx->num_sms;
        while (D.steps > 1 && n < most * step * D.steps) D.steps /= 2;  // every SM gets its blocks
        const long long g = std::min<long long>((n + step * D.steps - 1) / (step * D.steps), most);
        A.G.n = n;
        return launch_filter_with(A, grid, smem, lay, scratch, ctx->d_err, ctx->wait_cap, d_row_ids, capacity, d_count,
                                  d_sum, stream, &D, static_cast<int>(g));
    };
    if (plain && (variant == 1 || plain_loads_win(D, ids))) return run_plain();
    TQP_TRY(shape_filter(ctx, t, staged, bpr, ids, force, &A, &smem, &grid, &lay));
    const size_t used = ctx->used;
    void* scratch = arena_alloc(ctx, lay.bytes);
    if (!scratch && plain) {  // (its mask is not rounded up to whole tiles)
        ctx->used = used;
        return run_plain();
    }
    if (!scratch) return arena_oom(ctx, lay.bytes);
    return launch_filter_with(A, grid, smem, lay, scratch, ctx->d_err, ctx->wait_cap, d_row_ids, capacity, d_count,
                              d_sum, stream);
}

}  // namespace tqp

using namespace tqp;

extern "C" tqp_status tqp_filter(tqp_ctx* ctx, const tqp_table* t, const tqp_pred* preds, int32_t npreds,
                                 const tqp_expr* sum_expr, int64_t* d_sum, int32_t* d_row_ids, int64_t capacity,
                                 int64_t* d_count, void* stream) {
    clear_error();
    TQP_TRY(check_ctx(ctx));
    TQP_TRY(check_table(t, "tqp_filter"));
    if (!d_count) return fail(TQP_ERR_INVALID_ARG, "d_count is NULL");
    if ((sum_expr == nullptr) != (d_sum == nullptr))
        return fail(TQP_ERR_INVALID_ARG, "sum_expr and d_sum must both be set or both be NULL");
    if (d_row_ids && capacity < 0) return fail(TQP_ERR_INVALID_ARG, "capacity < 0");
    DeviceGuard g(ctx->device);
    if (!g.ok) return fail(TQP_ERR_CUDA, "cannot select device %d", ctx->device);
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::vector<int> cols;
    for (int i = 0; i < npreds && i < TQP_MAX_PREDS && preds; ++i) cols.push_back(preds[i].col);
    if (npreds == 0) expr_col_ids(sum_expr, cols);
    char key[96];
    snprintf(key, sizeof(key), "filter r%d b%d i%d s%d", rows_class(t->num_rows), row_bytes(t, cols),
             d_row_ids ? 1 : 0, sum_expr ? 1 : 0);
    auto run = [&]() {
        arena_reset(ctx);
        return launch_filter(ctx, t, preds, npreds, sum_expr, d_sum, d_row_ids, capacity, d_count, st, nullptr);
    };
    return tuned(ctx, key, st, npreds > 0 ? (kTuneVariant | kTuneV1Shapeless) : 0, run);
}

// ---- allocation-free variant (tqp_filter_noalloc) ------------------------------
// For callers that may not allocate device memory.  Its scratch is the
// file-scope array below (every device that loads the library holds it until
// exit): 256 bytes for the device error word, then the filter's own scratch
// layout (ticket, partial sums, block totals, selection mask) for at most
// TQP_NOALLOC_MAX_ROWS rows.  In host code `g_noalloc_scratch` names a host
// stand-in, not device memory, so its device address is looked up once per
// device (with that device current) and passed to the kernels.

namespace tqp {
constexpr size_t kNoallocErrBytes = 256;
constexpr size_t kNoallocScratchBytes = TQP_NOALLOC_SCRATCH_BYTES - kNoallocErrBytes;
}  // namespace tqp

static __device__ __align__(256) unsigned char g_noalloc_scratch[TQP_NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_noalloc_mu;
unsigned char* g_noalloc_addr[tqp::kMaxDevices] = {};

__global__ void k_noalloc_status(const int* err, int32_t* d_status) { *d_status = *err; }

// Device address of the scratch array on `device` (the caller made it current).
tqp_status noalloc_scratch(int device, unsigned char** out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[device]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_noalloc_addr[device] = static_cast<unsigned char*>(p);
    }
    *out = g_noalloc_addr[device];
    return TQP_OK;
}
}  // namespace

extern "C" tqp_status tqp_filter_noalloc(int device, const tqp_table* t, const tqp_pred* preds, int32_t npreds,
                                         const tqp_expr* sum_expr, int64_t* d_sum, int32_t* d_row_ids,
                                         int64_t capacity, int64_t* d_count, int32_t* d_status, void* stream) {
    clear_error();
    TQP_TRY(check_table(t, "tqp_filter_noalloc"));
    if (!d_count) return fail(TQP_ERR_INVALID_ARG, "d_count is NULL");
    if ((sum_expr == nullptr) != (d_sum == nullptr))
        return fail(TQP_ERR_INVALID_ARG, "sum_expr and d_sum must both be set or both be NULL");
    if (d_row_ids && capacity < 0) return fail(TQP_ERR_INVALID_ARG, "capacity < 0");
    if (t->num_rows > TQP_NOALLOC_MAX_ROWS)
        return fail(TQP_ERR_INVALID_ARG, "tqp_filter_noalloc handles at most %lld rows (got %lld); use tqp_filter",
                    (long long)TQP_NOALLOC_MAX_ROWS, (long long)t->num_rows);
    int ndev = 0;
    TQP_CUDA(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev || device >= kMaxDevices)
        return fail(TQP_ERR_INVALID_ARG, "device %d out of range", device);
    DeviceGuard g(device);
    if (!g.ok) return fail(TQP_ERR_CUDA, "cannot select device %d", device);
    unsigned char* base = nullptr;
    TQP_TRY(noalloc_scratch(device, &base));

    // a context-shaped description of the device; nothing here is allocated
    tqp_ctx dev_info{};
    dev_info.device = device;
    TQP_CUDA(cudaDeviceGetAttribute(&dev_info.num_sms, cudaDevAttrMultiProcessorCount, device));
    TQP_CUDA(cudaDeviceGetAttribute(&dev_info.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    dev_info.wait_cap = kDefaultWaitCap;

    FilterArgs A;
    size_t smem = 0;
    int grid = 0;
    FilterScratch lay;
    std::vector<int> staged;
    int bpr = 0;
    TQP_TRY(lower_filter(t, preds, npreds, sum_expr, &A, &staged, &bpr));
    TQP_TRY(shape_filter(&dev_info, t, staged, bpr, d_row_ids != nullptr, nullptr, &A, &smem, &grid, &lay));
    if (lay.bytes > kNoallocScratchBytes)
        return fail(TQP_ERR_INVALID_ARG, "tqp_filter_noalloc needs %zu scratch bytes, holds %zu", lay.bytes,
                    kNoallocScratchBytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int* err = reinterpret_cast<int*>(base);
    TQP_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));  // the array keeps the previous call's contents
    if (t->num_rows == 0) {
        TQP_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int64_t), st));
        if (d_sum) TQP_CUDA(cudaMemsetAsync(d_sum, 0, sizeof(int64_t), st));
    } else {
        TQP_TRY(launch_filter_with(A, grid, smem, lay, base + kNoallocErrBytes, err, kDefaultWaitCap, d_row_ids,
                                   capacity, d_count, d_sum, st));
    }
    if (d_status) {
        k_noalloc_status<<<1, 1, 0, st>>>(err, d_status);
        TQP_CUDA(cudaGetLastError());
    }
    return TQP_OK;
}
