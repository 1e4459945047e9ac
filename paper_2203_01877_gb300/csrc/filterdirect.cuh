// Filter scan with plain vector loads (paper Section 3.1: comparison mask, then
// the row ids of its set bits; Section 5.1: the sum of an expression over the
// passing rows), for at most kFdConds conditions and a sum that is a product of
// two affine factors. The conditions are sorted by column width, so that a step
// is straight code for its numbers of 64- and 32-bit ones.
//
// What bounds it is the memory system, so a warp step is short and many are in
// flight: 128 rows, four consecutive ones per lane, every condition column read
// with one load per lane (16 bytes for 32-bit columns, 32 for 64-bit ones), all
// issued before the first test, 32 warps per SM. The lanes' pass bits form four
// mask words. The sum's factors: where a step has many passing rows, its lanes
// read theirs with the same vector loads; the few rows of a selective query are
// queued per warp and evaluated 32 at a time, so that their load latency is paid
// once per 32 rows and not in every step. A warp takes up to kFdSteps consecutive
// steps and adds its count to its mask block with one atomic.
//
// Measured against the staged scan: 20M rows of which 96% pass, ids and sum, 557
// -> 125 us (this kernel 391 -> 96, the compaction 155 -> 22); 60M rows of which
// 1.8% pass 225 -> 222; the filters of a 512-plan batch 962 -> 562 (670 before the
// conditions were sorted by width). Evaluating a selective step's few rows at once
// instead of queueing them: 220 us instead of 201 for the 60M rows' kernel.
#pragma once

#include "bodies.cuh"
#include "partjoin.cuh"

namespace tqp {

constexpr int kFdThreads = 256;
constexpr int kFdMinBlocks = 4;
constexpr int kFdWide = 2;                         // conditions on 64-bit, 32-bit and 8-bit columns
constexpr int kFdWord = 3;
constexpr int kFdByte = 2;
constexpr int kFdConds = 4;                        // in all
constexpr int kFdStep = 4 * kWarp;                 // rows of a warp step
constexpr int kFdSteps = 4;                        // consecutive steps of a warp (a power of two): 60M rows take 222
                                                   // us a call, with 8 or 16 (a last wave mostly empty) 224 and 252,
                                                   // with 2 (an atomic per 256 rows) 234
constexpr int kFdDense = kFdStep / 4;              // passing rows of a step from which its lanes read their factors
constexpr int kFdQueue = kFdDense + kWarp;         // queued rows of a warp
constexpr int32_t kFdI64A32 = 16;                  // int64 column on a 32-byte boundary

// A row passes iff x - lo <= span in the column's arithmetic (32 bits for 8-
// and 32-bit columns); a negated range is the range of the other values.
struct FdCond {
    const unsigned char* p;
    int32_t a32;                  // 64-bit columns: on a 32-byte boundary
    int32_t pad;
    uint64_t lo;
    uint64_t span;
};

struct FilterDirectArgs {
    long long n;
    int32_t nwide, nword, nbyte;  // conditions of each width, in this order in `cond`
    int32_t has_sum;
    int32_t steps;                // of a warp: kFdSteps, fewer for small tables (a power of two)
    int32_t pad;
    FdCond cond[kFdConds];
    PjFactor f[2];                // the sum's factors (type: tqp_type, or kFdI64A32)
    uint32_t* mask;               // as in FilterArgs
    uint32_t* block_tot;
    unsigned long long* acc;      // [0] sum, [1] count, [2] finished blocks (zeroed)
    int64_t* d_count;
    int64_t* d_count2;
    int64_t* d_sum;
    int64_t capacity;
    int* err;
};

// Four consecutive rows' values: 64-bit ones in w[2 j], w[2 j + 1]; 32-bit ones
// in w[j]; 8-bit ones in the bytes of w[0].
struct FdRaw {
    uint32_t w[8];
};

// The lane's rows r .. r + 3 (all in the table; r a multiple of 4).
__device__ __forceinline__ void fd_load4(const unsigned char* p, int type, long long r, FdRaw& x) {
    if (type == TQP_I32) {
        const uint4 a = __ldcs(reinterpret_cast<const uint4*>(p + r * 4));
        x.w[0] = a.x;
        x.w[1] = a.y;
        x.w[2] = a.z;
        x.w[3] = a.w;
    } else if (type == kFdI64A32) {
        asm volatile("ld.global.cs.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3]), "=r"(x.w[4]), "=r"(x.w[5]), "=r"(x.w[6]),
                       "=r"(x.w[7])
                     : "l"(p + r * 8));
    } else if (type == TQP_I64) {
        const uint4 a = __ldcs(reinterpret_cast<const uint4*>(p + r * 8));
        const uint4 b = __ldcs(reinterpret_cast<const uint4*>(p + r * 8) + 1);
        x.w[0] = a.x;
        x.w[1] = a.y;
        x.w[2] = a.z;
        x.w[3] = a.w;
        x.w[4] = b.x;
        x.w[5] = b.y;
        x.w[6] = b.z;
        x.w[7] = b.w;
    } else {
        x.w[0] = __ldcs(reinterpret_cast<const unsigned int*>(p + r));
    }
}

// x[j] = the factor at row j of the raw values.
__device__ __forceinline__ void fd_factor(const PjFactor& f, const FdRaw& x, uint64_t (&v)[4]) {
    const uint64_t a = f.kind == kFacPlain || f.kind == kFacAdd ? 1u : (f.kind == kFacConst ? 0u : static_cast<uint64_t>(f.a));
    const uint64_t b = f.kind == kFacPlain ? 0u : static_cast<uint64_t>(f.b);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint64_t y = 0;
        if (f.kind != kFacConst) {
            if (f.type == TQP_I64 || f.type == kFdI64A32) y = x.w[2 * j] | (static_cast<uint64_t>(x.w[2 * j + 1]) << 32);
            else if (f.type == TQP_I32) y = static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(x.w[j])));
            else y = (x.w[0] >> (8 * j)) & 0xFFu;
        }
        v[j] = y * a + b;
    }
}

struct FdTotals {
    unsigned long long cnt = 0, sum = 0;
};

// The step's mask words: word k is the nibbles of lanes 8k .. 8k + 7.
__device__ __forceinline__ void fd_mask(const FilterDirectArgs& A, long long row0, int lane, uint32_t ok) {
    uint32_t v = ok << (4 * (lane & 7));
    v |= __shfl_xor_sync(0xffffffffu, v, 1);
    v |= __shfl_xor_sync(0xffffffffu, v, 2);
    v |= __shfl_xor_sync(0xffffffffu, v, 4);
    if ((lane & 7) == 0) A.mask[row0 / kWarp + lane / 8] = v;
}

// The sum's expression at one row.
__device__ __forceinline__ unsigned long long fd_eval(const FilterDirectArgs& A, long long r) {
    uint64_t x[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const PjFactor& f = A.f[k];
        x[k] = static_cast<uint64_t>(f.b);
        if (f.kind != kFacConst)
            x[k] += static_cast<uint64_t>(f.a) *
                    static_cast<uint64_t>(ldg_typed(f.p, f.type == kFdI64A32 ? TQP_I64 : f.type, r));
    }
    return x[0] * x[1];
}

// A warp's rows whose expression is still to be evaluated (fewer than kWarp between steps).
struct FdQueue {
    uint32_t* row;
    int n;
};

// Passing rows of the lane in a step that lies in the table; NW conditions on
// 64-bit columns and NN on 32-bit ones.
template <int NW, int NN>
__device__ __forceinline__ uint32_t fd_step(const FilterDirectArgs& A, long long row0, int lane, unsigned long long& sum,
                                            FdQueue& Q) {
    const long long r = row0 + 4 * lane;
    FdRaw wide[NW ? NW : 1], word[NN ? NN : 1];
    uint32_t byte[kFdByte];
#pragma unroll
    for (int c = 0; c < NW; ++c) fd_load4(A.cond[c].p, A.cond[c].a32 ? kFdI64A32 : TQP_I64, r, wide[c]);
#pragma unroll
    for (int c = 0; c < NN; ++c) fd_load4(A.cond[NW + c].p, TQP_I32, r, word[c]);
#pragma unroll
    for (int c = 0; c < kFdByte; ++c)
        if (c < A.nbyte) byte[c] = __ldcs(reinterpret_cast<const unsigned int*>(A.cond[NW + NN + c].p + r));
    bool p[4] = {true, true, true, true};
#pragma unroll
    for (int c = 0; c < NW; ++c) {
        const FdCond& f = A.cond[c];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            p[j] = p[j] && (wide[c].w[2 * j] | (static_cast<uint64_t>(wide[c].w[2 * j + 1]) << 32)) - f.lo <= f.span;
    }
#pragma unroll
    for (int c = 0; c < NN; ++c) {
        const uint32_t lo = static_cast<uint32_t>(A.cond[NW + c].lo), span = static_cast<uint32_t>(A.cond[NW + c].span);
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = p[j] && word[c].w[j] - lo <= span;
    }
#pragma unroll
    for (int c = 0; c < kFdByte; ++c) {
        if (c >= A.nbyte) break;
        const uint32_t lo = static_cast<uint32_t>(A.cond[NW + NN + c].lo);
        const uint32_t span = static_cast<uint32_t>(A.cond[NW + NN + c].span);
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = p[j] && ((byte[c] >> (8 * j)) & 0xFFu) - lo <= span;
    }
    const uint32_t ok = static_cast<uint32_t>(p[0]) | static_cast<uint32_t>(p[1]) << 1 | static_cast<uint32_t>(p[2]) << 2 |
                        static_cast<uint32_t>(p[3]) << 3;
    if (A.mask) fd_mask(A, row0, lane, ok);
    const uint32_t cnt = __popc(ok);
    if (!A.has_sum) return cnt;
    const uint32_t all = __reduce_add_sync(0xffffffffu, cnt);
    if (all >= kFdDense) {
        if (!ok) return cnt;
        FdRaw y[2];
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (A.f[k].kind != kFacConst) fd_load4(A.f[k].p, A.f[k].type, r, y[k]);
        uint64_t v0[4], v1[4];
        fd_factor(A.f[0], y[0], v0);
        fd_factor(A.f[1], y[1], v1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((ok >> j) & 1u) sum += v0[j] * v1[j];
    } else if (all) {
        const uint32_t lt = lanemask_lt();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t m = __ballot_sync(0xffffffffu, (ok >> j) & 1u);
            if ((ok >> j) & 1u) Q.row[Q.n + __popc(m & lt)] = static_cast<uint32_t>(r + j);
            Q.n += __popc(m);
        }
        __syncwarp();
        if (Q.n >= kWarp) {
            sum += fd_eval(A, Q.row[Q.n - kWarp + lane]);
            Q.n -= kWarp;
            __syncwarp();
        }
    }
    return cnt;
}

// The table's last step, row by row: pass bits of rows r .. r + 3.
static __device__ __noinline__ uint32_t fd_tail(const FilterDirectArgs& A, long long r, unsigned long long* sum) {
    uint32_t ok = 0;
    for (int j = 0; j < 4 && r + j < A.n; ++j) {
        bool pass = true;
        for (int c = 0; c < A.nwide + A.nword + A.nbyte; ++c) {
            const FdCond& f = A.cond[c];
            const int type = c < A.nwide ? TQP_I64 : (c < A.nwide + A.nword ? TQP_I32 : TQP_U8);
            const uint64_t d = static_cast<uint64_t>(ldg_typed(f.p, type, r + j)) - f.lo;
            pass = pass && (type == TQP_I64 ? d <= f.span : static_cast<uint32_t>(d) <= static_cast<uint32_t>(f.span));
        }
        if (!pass) continue;
        ok |= 1u << j;
        if (A.has_sum) *sum += fd_eval(A, r + j);
    }
    return ok;
}

template <int NW, int NN>
__device__ __forceinline__ void fd_loop(const FilterDirectArgs& A, long long vb, long long vg, int lane, int w,
                                        uint32_t* queue, FdTotals& T) {
    FdQueue Q{queue, 0};
    const long long seg = static_cast<long long>(A.steps) * kFdStep;  // a divisor of kCompactRows
    const long long stride = vg * (kFdThreads / kWarp) * seg;
    for (long long s0 = (vb * (kFdThreads / kWarp) + w) * seg; s0 < A.n; s0 += stride) {
        uint32_t c = 0;
        long long r0 = s0;
        const long long s1 = s0 + seg < A.n ? s0 + seg : A.n;
#pragma unroll 1
        for (; r0 + kFdStep <= s1; r0 += kFdStep) c += fd_step<NW, NN>(A, r0, lane, T.sum, Q);
        if (r0 < s1) {
            unsigned long long t = 0;
            const uint32_t ok = fd_tail(A, r0 + 4 * lane, &t);
            T.sum += t;
            c += __popc(ok);
            if (A.mask) fd_mask(A, r0, lane, ok);
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) {
            T.cnt += c;
            if (A.mask && c) atomicAdd(&A.block_tot[s0 / kCompactRows], c);
        }
    }
    if (lane < Q.n) T.sum += fd_eval(A, Q.row[lane]);
}

// Block vb of vg working on this filter.
static __device__ __forceinline__ void filter_direct_block(const FilterDirectArgs& A, long long vb, long long vg) {
    __shared__ unsigned long long red[2][kFdThreads / kWarp];
    __shared__ uint32_t queue[kFdThreads / kWarp][kFdQueue];  // (one for all the forms of fd_loop)
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    FdTotals T;
    switch (A.nwide * (kFdWord + 1) + A.nword) {
        case 0: fd_loop<0, 0>(A, vb, vg, lane, w, queue[w], T); break;
        case 1: fd_loop<0, 1>(A, vb, vg, lane, w, queue[w], T); break;
        case 2: fd_loop<0, 2>(A, vb, vg, lane, w, queue[w], T); break;
        case 3: fd_loop<0, 3>(A, vb, vg, lane, w, queue[w], T); break;
        case 4: fd_loop<1, 0>(A, vb, vg, lane, w, queue[w], T); break;
        case 5: fd_loop<1, 1>(A, vb, vg, lane, w, queue[w], T); break;
        case 6: fd_loop<1, 2>(A, vb, vg, lane, w, queue[w], T); break;
        case 7: fd_loop<1, 3>(A, vb, vg, lane, w, queue[w], T); break;
        case 8: fd_loop<2, 0>(A, vb, vg, lane, w, queue[w], T); break;
        case 9: fd_loop<2, 1>(A, vb, vg, lane, w, queue[w], T); break;
        default: fd_loop<2, 2>(A, vb, vg, lane, w, queue[w], T); break;  // (at most kFdConds in all)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) T.sum += __shfl_xor_sync(0xffffffffu, T.sum, o);
    if (lane == 0) {
        red[0][w] = T.sum;
        red[1][w] = T.cnt;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    unsigned long long t[2] = {0, 0};
    for (int i = 0; i < kFdThreads / kWarp; ++i)
        for (int k = 0; k < 2; ++k) t[k] += red[k][i];
    for (int k = 0; k < 2; ++k)
        if (t[k]) atomicAdd(&A.acc[k], t[k]);
    __threadfence();
    if (atomicAdd(&A.acc[2], 1ULL) != static_cast<unsigned long long>(vg) - 1ULL) return;
    __threadfence();
    const unsigned long long sum = atomicAdd(&A.acc[0], 0ULL), cnt = atomicAdd(&A.acc[1], 0ULL);
    *A.d_count = static_cast<int64_t>(cnt);
    if (A.d_count2) *A.d_count2 = static_cast<int64_t>(cnt);
    if (A.d_sum) *A.d_sum = static_cast<int64_t>(sum);
    if (A.mask && static_cast<long long>(cnt) > A.capacity) latch_error(A.err, TQP_ERR_CAPACITY);
}

// Host (filter.cu): lower a filter to this form; false outside its shapes.
bool lower_filter_direct(const tqp_table* t, const FilterArgs& F, FilterDirectArgs* A);

}  // namespace tqp
