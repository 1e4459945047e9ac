// Group-by over key columns of small range (the aggregation of paper Section
// 5.4 without a hash table and without a sort): when the key columns' ranges
// multiply to no more entries than the group table holds, a row's entry is its
// mixed-radix index sum (x_i - min_i) * stride_i, so one pass over the rows
// adds each to its entry, and the entries in index order are the groups in key
// order.  Decided on the device from the key ranges; the hash kernels return at
// once when it applies, and these do when it does not.
//
//   k_group_range   clears the entries and the hash path's table; [min, max] of
//                   every key column; the last block writes the plan. A sample of
//                   256 rows whose ranges do not fit leaves the pass out, so that
//                   scattered keys pay for two short launches
//   k_group_clear   (tables above kGrClearBytes) the clearing, of what is used only
//   k_group_agg     few entries: a table per CTA in shared memory, flushed once;
//                   the rest: one reduction instruction per row into L2, the words
//                   of an entry on neighbouring lanes (probeagg.cuh; k_group_l2
//                   from kGrSplitRows rows on)
//   the hash path's output kernels: used entries -> output rows
//
// What bounds the L2 form is the L2's reduction rate (about 206 G sector
// operations per second), not the 12 bytes a row streams; the rows of
// an entry that is hot in a warp are added up first, since reductions on one
// 128-byte line serialise.
//
// Measured (60M rows, one int32 key, SUM and COUNT; hash path -> this): 1.5M
// groups 3324 -> 473 us, of them k_group_l2 375 and the range pass 47; 60K groups
// 3240 -> 495; 10K groups (shared memory) 2358 -> 308. 100K rows, 1000 groups:
// 124 -> 37. Entries beyond shared memory go to L2 from about 17K (one sum). Keys
// the sample finds scattered: 60M rows 3348 -> 3390, 6M rows 459 -> 440, 10K rows
// 119 -> 121 (with the whole range pass and five more launches 3473, 465 and 141).
#pragma once

#include "groupdirect.cuh"
#include "probeagg.cuh"

namespace tqp {

constexpr int kGrVals = 3;                      // sums
constexpr int kGrThreads = 768;                 // one CTA per SM: 24 warps at 85 registers
constexpr int kGrSmemBytes = 208 * 1024;
constexpr long long kGrRowsPerEntry = 256;      // of a table in shared memory, at least
constexpr int kGrEmitThreads = 256;
constexpr int kGrEmitPer = 4096;                // entries of a block of the output kernels
constexpr long long kGrMaxEntries = 1LL << 24;  // (every output block adds up the blocks' counts)
constexpr long long kGrSplitRows = 1LL << 23;   // rows from which the L2 form has its own kernel (beside it L1 stays large)
constexpr size_t kGrClearBytes = 2 << 20;       // tables up to this are cleared before their range is known
constexpr long long kGrClearPer = 16 << 10;     // bytes of a block

struct GroupRangePlan {
    unsigned long long kmeta[2 * kDirKeys];  // as GroupDirectArgs::kmeta (zeroed)
    unsigned int done;                       // finished range blocks (zeroed)
    int32_t on;                              // the entries fit: this path runs, the hash path does not
    int32_t smem;                            // the entries fit shared memory
    int32_t pad;
    long long entries;
    long long lo[kDirKeys];
    unsigned long long range[kDirKeys];
    unsigned int stride[kDirKeys];
};

struct GroupRangeArgs {
    long long n;
    int32_t ncond;
    int32_t ngc;
    int32_t nval;
    int32_t pad;
    PjCond cond[TQP_MAX_PREDS];
    PjCol key[kDirKeys];
    PjFactor f[kGrVals][2];
    GroupRangePlan* plan;
    unsigned long long* acc;  // entries of nval + 1 words (count first)
    long long max_entries;
};

// Clears the entries and keys of the hash path's table (`words` accumulator words, the count of distinct keys behind them).
__device__ __forceinline__ void group_clear(const GroupSpec& S, long long words, bool keys) {
    const long long tid = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    const long long nth = static_cast<long long>(gridDim.x) * blockDim.x;
    ulonglong2* p = reinterpret_cast<ulonglong2*>(S.acc);
    for (long long i = tid; i < words / 2; i += nth) p[i] = make_ulonglong2(0, 0);
    if (tid == 0 && words % 2) S.acc[words - 1] = 0;
    if (!keys) return;
    for (long long i = tid; i <= S.cap; i += nth) S.keys[i] = kEmptyKey;
}

// d *= the entries of one more key column with (encoded) range [mn, mx]; false when they are more than `most`.
__device__ __forceinline__ bool gr_widen(unsigned long long& d, unsigned long long mn, unsigned long long mx,
                                         unsigned long long most) {
    if (mx - mn >= most) return false;
    d *= mx - mn + 1;  // (both factors below 2^25)
    return d <= most;
}

// Whether the ranges of 256 rows spread over the table fit the entries (the same in every block).
__device__ __forceinline__ bool gr_sample_fits(const GroupRangeArgs& A) {
    __shared__ unsigned long long part[2][kDirThreads / kWarp];
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const long long r = static_cast<long long>(static_cast<unsigned long long>(A.n) * threadIdx.x / kDirThreads);
    unsigned long long d = 1;
    bool fits = true;
    for (int i = 0; i < A.ngc; ++i) {
        unsigned long long mx = 0, mn = 0;
        dir_enc_update(ldg_typed(A.key[i].p, A.key[i].type, r), mx, mn);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, mx, o), b = __shfl_xor_sync(0xffffffffu, mn, o);
            mx = a > mx ? a : mx;
            mn = b > mn ? b : mn;
        }
        if (lane == 0) {
            part[0][w] = mn;
            part[1][w] = mx;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kDirThreads / kWarp; ++k) {
            mn = part[0][k] > mn ? part[0][k] : mn;
            mx = part[1][k] > mx ? part[1][k] : mx;
        }
        __syncthreads();
        fits = fits && gr_widen(d, ~mn, mx, static_cast<unsigned long long>(A.max_entries));
    }
    return fits;
}

__device__ __forceinline__ void group_range_block(const GroupRangeArgs& A) {
    GroupRangePlan* P = A.plan;
    if (!gr_sample_fits(A)) return;  // (the plan stays off)
    group_direct_range_block(A, P->kmeta, nullptr, blockIdx.x, gridDim.x);
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(&P->done, 1u) != gridDim.x - 1) return;
    __threadfence();
    unsigned long long d = 1;
    bool on = true;
    for (int i = A.ngc - 1; i >= 0; --i) {
        const unsigned long long mn = ~atomicAdd(&P->kmeta[2 * i], 0ULL), mx = atomicAdd(&P->kmeta[2 * i + 1], 0ULL);
        P->lo[i] = static_cast<long long>(mn ^ 0x8000000000000000ull);
        P->range[i] = mx - mn + 1;
        P->stride[i] = static_cast<unsigned int>(d);
        on = on && gr_widen(d, mn, mx, static_cast<unsigned long long>(A.max_entries));
        if (!on) d = 1;
    }
    P->entries = static_cast<long long>(d);
    // a CTA's table must be worth clearing and flushing: more rows than entries
    P->smem = d * (4 + 8 * A.nval) <= kGrSmemBytes && A.n >= kGrRowsPerEntry * static_cast<long long>(d);
    P->on = on;
}

// The entry of each of the lane's four rows (kPaNone: not a passing row).
template <bool kFull>
__device__ __forceinline__ void gr_entries(const GroupRangeArgs& A, const GroupRangePlan& P, long long r0, int lane,
                                           uint32_t in, uint32_t (&e)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) e[j] = 0;
    for (int i = 0; i < A.ngc; ++i) {
        int64_t x[4];
        pa_col<kFull>(A.key[i].p, A.key[i].type, r0, lane, in, x);
        const uint32_t lo = static_cast<uint32_t>(P.lo[i]), st = P.stride[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] += (static_cast<uint32_t>(x[j]) - lo) * st;
    }
}

template <bool kFull, int W>
__device__ __forceinline__ void gr_values(const GroupRangeArgs& A, long long r0, int lane, uint32_t in,
                                          int64_t (&v)[3][4]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[a][j] = 0;
        if (a + 1 < W) pa_prod<kFull>(A.f[a], r0, lane, in, v[a]);
    }
}

__device__ __forceinline__ uint32_t gr_in(const GroupRangeArgs& A, long long r0, int lane) {
    uint32_t in = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) in |= static_cast<uint32_t>(pa_row(r0, lane, j) < A.n) << j;
    return in;
}

// ---- entries in L2 -------------------------------------------------------------

template <bool kFull, int W>
__device__ __forceinline__ void gr_l2_step(const GroupRangeArgs& A, const GroupRangePlan& P, long long r0, int lane,
                                           uint32_t& hot) {
    const uint32_t in = kFull ? 0xFu : gr_in(A, r0, lane);
    uint32_t e[4];
    int64_t v[3][4];
    gr_entries<kFull>(A, P, r0, lane, in, e);
    gr_values<kFull, W>(A, r0, lane, in, v);
    const uint32_t ok = pa_conds<kFull>(A, r0, lane, in);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (!((ok >> j) & 1u)) e[j] = kPaNone;
    pa_combine<W>(A.acc, W, e, v[0], v[1], v[2], lane, hot);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned long long x[3] = {static_cast<unsigned long long>(v[0][j]),
                                         static_cast<unsigned long long>(v[1][j]),
                                         static_cast<unsigned long long>(v[2][j])};
        pa_red<W>(A.acc, W, e[j], x, lane);
    }
}

template <int W, int kThreads>
__device__ __forceinline__ void gr_l2_loop(const GroupRangeArgs& A, const GroupRangePlan& P) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const long long stride = static_cast<long long>(gridDim.x) * (kThreads / kWarp) * kPaStep;
    uint32_t hot = kPaNone;
    for (long long r0 = (static_cast<long long>(blockIdx.x) * (kThreads / kWarp) + w) * kPaStep; r0 < A.n;
         r0 += stride) {
        if (r0 + kPaStep <= A.n) gr_l2_step<true, W>(A, P, r0, lane, hot);
        else gr_l2_step<false, W>(A, P, r0, lane, hot);
    }
}

template <int kThreads>
__device__ __forceinline__ void group_l2_block(const GroupRangeArgs& A, const GroupRangePlan& P) {
    switch (A.nval) {
        case 0: gr_l2_loop<1, kThreads>(A, P); break;
        case 1: gr_l2_loop<2, kThreads>(A, P); break;
        case 2: gr_l2_loop<3, kThreads>(A, P); break;
        default: gr_l2_loop<4, kThreads>(A, P); break;
    }
}

// ---- entries in shared memory ----------------------------------------------------

template <bool kFull>
__device__ __forceinline__ void gr_smem_step(const GroupRangeArgs& A, const GroupRangePlan& P, uint32_t* tab, long long r0,
                                             int lane) {
    const uint32_t in = kFull ? 0xFu : gr_in(A, r0, lane);
    uint32_t e[4];
    gr_entries<kFull>(A, P, r0, lane, in, e);
    const uint32_t ok = pa_conds<kFull>(A, r0, lane, in);
    const uint32_t D = static_cast<uint32_t>(P.entries);
    int64_t v[3][4];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (a < A.nval) pa_prod<kFull>(A.f[a], r0, lane, in, v[a]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned long long x[3] = {static_cast<unsigned long long>(v[0][j]),
                                         static_cast<unsigned long long>(v[1][j]),
                                         static_cast<unsigned long long>(v[2][j])};
        if ((ok >> j) & 1u) pa_smem_add(tab, D, e[j], A.nval, x);
    }
}

__device__ __forceinline__ void group_smem_block(const GroupRangeArgs& A, const GroupRangePlan& P, uint32_t* tab) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const uint32_t D = static_cast<uint32_t>(P.entries);
    for (uint32_t i = threadIdx.x; i < D * (1 + 2 * A.nval); i += kGrThreads) tab[i] = 0;
    __syncthreads();
    const long long stride = static_cast<long long>(gridDim.x) * (kGrThreads / kWarp) * kPaStep;
    for (long long r0 = (static_cast<long long>(blockIdx.x) * (kGrThreads / kWarp) + w) * kPaStep; r0 < A.n;
         r0 += stride) {
        if (r0 + kPaStep <= A.n) gr_smem_step<true>(A, P, tab, r0, lane);
        else gr_smem_step<false>(A, P, tab, r0, lane);
    }
    __syncthreads();
    pa_smem_flush(tab, D, A.nval, A.acc, A.nval + 1);
}

// ---- output ----------------------------------------------------------------------

// The packed key of entry e.
__device__ __forceinline__ uint64_t gr_key(const GroupRangePlan* plan, const GroupSpec& S, long long e) {
    uint64_t key = 0;
    for (int i = 0; i < S.ngc; ++i) {
        const uint32_t d = static_cast<uint32_t>(e) / plan->stride[i] % static_cast<uint32_t>(plan->range[i]);
        const uint64_t c = enc_key(plan->lo[i] + d, S.key_bits[i]);
        key = S.key_bits[i] == 64 ? c : ((key << S.key_bits[i]) | c);
    }
    return key;
}

// The groups of at most kSmallCap + 1 entries, by one block of kFinThreads. (A
// call: in line it costs the hash path's output 1 us.)
static __device__ __noinline__ void group_rows_small(const GroupRangePlan* plan, const GroupSpec& S, const GroupOut& O) {
    constexpr int kPer = kSmallCap / kFinThreads + 1;
    __shared__ uint32_t wcnt[kFinThreads / kWarp];
    const long long D = plan->entries;
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    uint32_t used = 0;
    int G = 0;
#pragma unroll
    for (int s = 0; s < kPer; ++s) {
        const long long e = s * kFinThreads + threadIdx.x;
        const bool u = e < D && S.acc[e * S.nacc] != 0;
        used |= static_cast<uint32_t>(u) << s;
        G += __syncthreads_count(u);
    }
    if (G > S.max_groups || G > O.capacity) {
        if (threadIdx.x == 0) {
            *O.num_groups = -1;
            latch_error(O.err, TQP_ERR_CAPACITY);
        }
        return;
    }
    if (threadIdx.x == 0) *O.num_groups = G;
    int first = 0;
    for (int s = 0; s < kPer; ++s) {
        const bool u = (used >> s) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, u);
        if (lane == 0) wcnt[w] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
        for (int k = 0; k < kFinThreads / kWarp; ++k) {
            before += k < w ? wcnt[k] : 0;
            all += wcnt[k];
        }
        __syncthreads();
        const long long e = s * kFinThreads + threadIdx.x;
        if (u) emit_group(S, O, first + before + __popc(m & lanemask_lt()), gr_key(plan, S, e), e);
        first += all;
    }
}

// The used entries of output block b.
__device__ __forceinline__ void group_count_block(const GroupRangePlan* plan, const GroupSpec& S, uint32_t* counts, int b) {
    const long long e0 = static_cast<long long>(b) * kGrEmitPer, D = plan->entries;
    int c = 0;
    for (int s = 0; s < kGrEmitPer / kGrEmitThreads; ++s) {
        const long long e = e0 + s * kGrEmitThreads + threadIdx.x;
        c += __syncthreads_count(e < D && S.acc[e * S.nacc] != 0);
    }
    if (threadIdx.x == 0) counts[b] = static_cast<uint32_t>(c);
}

__device__ __forceinline__ int gr_blocks(const GroupRangePlan* plan) {
    return static_cast<int>((plan->entries + kGrEmitPer - 1) / kGrEmitPer);
}

// The groups of output block b; false when there are too many of them.
__device__ __forceinline__ bool group_rows_block(const GroupRangePlan* plan, const GroupSpec& S, const GroupOut& O,
                                                 const uint32_t* counts, int b) {
    __shared__ unsigned long long sums[2];
    __shared__ uint32_t wcnt[kGrEmitPer / kWarp];
    const long long D = plan->entries;
    const int nb = gr_blocks(plan);
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    if (threadIdx.x < 2) sums[threadIdx.x] = 0;
    __syncthreads();
    // groups in the blocks before this one, and in all
    unsigned long long before = 0, total = 0;
    for (int i = threadIdx.x; i < nb; i += kGrEmitThreads) {
        const uint32_t c = counts[i];
        total += c;
        if (i < b) before += c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    if (lane == 0) {
        atomicAdd(&sums[0], before);
        atomicAdd(&sums[1], total);
    }
    __syncthreads();
    const long long G = static_cast<long long>(sums[1]);
    if (G > S.max_groups || G > O.capacity) {
        if (b == 0 && threadIdx.x == 0) {
            *O.num_groups = -1;
            latch_error(O.err, TQP_ERR_CAPACITY);
        }
        return false;
    }
    if (b == 0 && threadIdx.x == 0) *O.num_groups = G;
    const long long e0 = static_cast<long long>(b) * kGrEmitPer;
    uint32_t used = 0;  // of the thread's entries e0 + 256 s + threadIdx.x
#pragma unroll
    for (int s = 0; s < kGrEmitPer / kGrEmitThreads; ++s) {
        const long long e = e0 + s * kGrEmitThreads + threadIdx.x;
        const bool u = e < D && S.acc[e * S.nacc] != 0;
        const uint32_t m = __ballot_sync(0xffffffffu, u);
        used |= static_cast<uint32_t>(u) << s;
        if (lane == 0) wcnt[s * (kGrEmitThreads / kWarp) + w] = __popc(m);
    }
    __syncthreads();
    if (w == 0) {  // exclusive scan of the 128 warp counts, four per lane
        uint32_t c[4], t = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c[k] = t;
            t += wcnt[4 * lane + k];
        }
        uint32_t incl = t;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) wcnt[4 * lane + k] = incl - t + c[k];
    }
    __syncthreads();
    for (int s = 0; s < kGrEmitPer / kGrEmitThreads; ++s) {
        const bool u = (used >> s) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, u);
        if (!u) continue;
        const long long e = e0 + s * kGrEmitThreads + threadIdx.x;
        emit_group(S, O, static_cast<long long>(sums[0]) + wcnt[s * (kGrEmitThreads / kWarp) + w] +
                             __popc(m & lanemask_lt()), gr_key(plan, S, e), e);
    }
    return true;
}
static_assert(kGrEmitPer / kWarp == 4 * kWarp, "one warp scans the warp counts");

}  // namespace tqp
