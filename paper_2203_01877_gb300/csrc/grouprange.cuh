// Group-by over key columns of small range (the aggregation of paper Section
// 5.4 without a hash table and without a sort): when the key columns' ranges
// multiply to no more entries than the group table holds, a row's entry is its
// mixed-radix index sum (x_i - min_i) * stride_i, so one pass over the rows
// adds each to its entry, and the entries in index order are the groups in key
// order.  Decided on the device from the key ranges; the hash kernels return at
// once when it applies, and these do when it does not.
//
//   k_group_range   [min, max] of every key column; the last block writes the plan
//   k_group_clear   the entries (or, for the hash path, its table)
//   k_group_smem    few entries: a table per CTA in shared memory, flushed once
//   k_group_l2      the rest: one reduction instruction per row into L2, the
//                   words of an entry on neighbouring lanes (probeagg.cuh)
//   k_group_count, k_group_rows   used entries -> output rows
//
// What bounds k_group_l2 is the L2's reduction rate (about 206 G sector
// operations per second), not the 12 bytes a row streams; the rows of
// an entry that is hot in a warp are added up first, since reductions on one
// 128-byte line serialise.
//
// Measured (60M rows, one int32 key, SUM and COUNT; hash path -> this): 1.5M
// groups 3206 -> 493 us, of them k_group_l2 375 and the range pass 47; 60K groups
// 2978 -> 531; 10K groups (shared memory) 2257 -> 311; 1K groups 3170 -> 284.
// 100K rows, 1000 groups: 113 -> 47.  Entries beyond shared memory go to L2 from
// about 17K (one sum): 20K groups take 601 us there, more than 10K in shared
// memory, less than the hash path's 2284.
#pragma once

#include "groupdirect.cuh"
#include "probeagg.cuh"

namespace tqp {

constexpr int kGrVals = 3;                      // sums
constexpr int kGrSmemThreads = 768;             // one CTA per SM: 24 warps at 85 registers
constexpr int kGrSmemBytes = 208 * 1024;
constexpr int kGrEmitThreads = 256;
constexpr int kGrEmitPer = 4096;                // entries of a block of the output kernels
constexpr long long kGrMaxEntries = 1LL << 24;  // (every output block adds up the blocks' counts)

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

__device__ __forceinline__ void group_range_block(const GroupRangeArgs& A) {
    GroupRangePlan* P = A.plan;
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
        on = on && mx - mn < static_cast<unsigned long long>(A.max_entries);
        const unsigned long long r = on ? mx - mn + 1 : 1;
        P->range[i] = r;
        P->stride[i] = static_cast<unsigned int>(d);
        d *= r;  // (both factors below 2^25)
        on = on && d <= static_cast<unsigned long long>(A.max_entries);
        if (!on) d = 1;
    }
    P->entries = static_cast<long long>(d);
    // a CTA's table must be worth clearing and flushing: more rows than entries
    P->smem = d * (4 + 8 * A.nval) <= kGrSmemBytes && A.n >= 256 * static_cast<long long>(d);
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

template <int W>
__device__ __forceinline__ void gr_l2_loop(const GroupRangeArgs& A, const GroupRangePlan& P) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const long long stride = static_cast<long long>(gridDim.x) * (kPaThreads / kWarp) * kPaStep;
    uint32_t hot = kPaNone;
    for (long long r0 = (static_cast<long long>(blockIdx.x) * (kPaThreads / kWarp) + w) * kPaStep; r0 < A.n;
         r0 += stride) {
        if (r0 + kPaStep <= A.n) gr_l2_step<true, W>(A, P, r0, lane, hot);
        else gr_l2_step<false, W>(A, P, r0, lane, hot);
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

__device__ __forceinline__ void group_smem_block(const GroupRangeArgs& A, uint32_t* tab) {
    const GroupRangePlan P = *A.plan;
    if (!P.on || !P.smem) return;
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const uint32_t D = static_cast<uint32_t>(P.entries);
    for (uint32_t i = threadIdx.x; i < D * (1 + 2 * A.nval); i += kGrSmemThreads) tab[i] = 0;
    __syncthreads();
    const long long stride = static_cast<long long>(gridDim.x) * (kGrSmemThreads / kWarp) * kPaStep;
    for (long long r0 = (static_cast<long long>(blockIdx.x) * (kGrSmemThreads / kWarp) + w) * kPaStep; r0 < A.n;
         r0 += stride) {
        if (r0 + kPaStep <= A.n) gr_smem_step<true>(A, P, tab, r0, lane);
        else gr_smem_step<false>(A, P, tab, r0, lane);
    }
    __syncthreads();
    pa_smem_flush(tab, D, A.nval, A.acc, A.nval + 1);
}

// ---- output ----------------------------------------------------------------------

__device__ __forceinline__ void group_rows_block(const GroupRangePlan* plan, const GroupSpec& S, const GroupOut& O,
                                                 const uint32_t* counts) {
    __shared__ unsigned long long sums[2];
    __shared__ uint32_t wcnt[kGrEmitPer / kWarp];
    if (!plan->on) return;
    const long long D = plan->entries;
    const int nb = static_cast<int>((D + kGrEmitPer - 1) / kGrEmitPer);
    if (static_cast<int>(blockIdx.x) >= nb) return;
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    if (threadIdx.x < 2) sums[threadIdx.x] = 0;
    __syncthreads();
    // groups in the blocks before this one, and in all
    unsigned long long before = 0, total = 0;
    for (int i = threadIdx.x; i < nb; i += kGrEmitThreads) {
        const uint32_t c = counts[i];
        total += c;
        if (i < static_cast<int>(blockIdx.x)) before += c;
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
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *O.num_groups = -1;
            latch_error(O.err, TQP_ERR_CAPACITY);
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *O.num_groups = G;
    const long long e0 = static_cast<long long>(blockIdx.x) * kGrEmitPer;
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
        uint64_t key = 0;
        for (int i = 0; i < S.ngc; ++i) {
            const uint32_t d = static_cast<uint32_t>(e) / plan->stride[i] % static_cast<uint32_t>(plan->range[i]);
            const uint64_t c = enc_key(plan->lo[i] + d, S.key_bits[i]);
            key = S.key_bits[i] == 64 ? c : ((key << S.key_bits[i]) | c);
        }
        emit_group(S, O, static_cast<long long>(sums[0]) + wcnt[s * (kGrEmitThreads / kWarp) + w] +
                             __popc(m & lanemask_lt()), key, e);
    }
}
static_assert(kGrEmitPer / kWarp == 4 * kWarp, "one warp scans the warp counts");

}  // namespace tqp
