// Joined aggregation by a probe with plain loads: filter, probe and aggregate
// the fact rows of a join plan (the join -> group-by of paper Sections 5.3 and
// 5.4, never materialised), for the closed-form shapes PlanJoinBody::step_fast
// covers -- every condition, the foreign key and the factors of at most two
// group sums and the ungrouped sum are plain columns.
//
// What bounds it is the L2: a probe row costs one random gather (hashed
// tables; 290 G/s measured) and one random reduction of its entry (206 G/s),
// against 12 bytes streamed, so the kernel wants many warps in flight and few
// L2 operations per row:
//   * no staging: a warp takes 128 consecutive rows per step with vector
//     loads, and 24 to 32 warps per SM hide the latency of loads, gathers and
//     shuffles (the staged body ran one CTA of 9 warps per SM at 142 registers
//     and was latency-bound);
//   * the words of a row's entry (count and sums) go out in ONE reduction
//     instruction with neighbouring lanes holding neighbouring words: an L2
//     reduction costs per 32-byte sector an instruction touches, not per word
//     (60M random 16-byte entries: 585 us with a reduction per word, 291 us
//     with a lane pair; 32-byte entries: 1166 against 464 us);
//   * reductions on one 128-byte line serialise (2.5 ns each), so entries that
//     fit a CTA's shared memory are accumulated there and flushed once, and
//     the rows of an entry that is hot in a warp are added up before they go.
// Lane l of a step handles rows 2l, 2l + 1, 64 + 2l and 64 + 2l + 1: loads of
// 1-, 4- and 8-byte columns are all contiguous across the warp.
#pragma once

#include "group.cuh"
#include "join.cuh"
#include "partjoin.cuh"

namespace tqp {

constexpr int kPaThreads = 256;
constexpr int kPaMinBlocks = 3;      // 24 warps per SM: 85 registers
constexpr int kPaStep = 4 * kWarp;   // rows of a warp step
constexpr int kPaVals = 2;           // group sums
constexpr uint32_t kPaNone = 0xFFFFFFFFu;
constexpr int kPaSmemBytes = 64 * 1024;  // the CTA's entries: a 32-bit count and 64-bit sums each

struct ProbeAggArgs {
    long long n;              // fact rows
    int32_t ncond;
    int32_t nval;             // group sums (<= kPaVals)
    int32_t has_sum;          // ungrouped SUM over joined rows
    int32_t nk;               // words per key-first entry
    PjCond cond[TQP_MAX_PREDS];  // clamped to the column type (lower_fast)
    PjCol fk;
    PjFactor f[kPaVals][2];   // group sum a = f[a][0] * f[a][1]
    PjFactor fs[2];           // the ungrouped sum
    JoinHT H;                 // cap < 2^31
    const uint32_t* next;     // chained build: next dim row of the same key
    const uint32_t* dgs;      // dim row -> dense group id; nullptr: no aggregation
    const long long* d_groups; // groups (entries of gacc)
    unsigned long long* gacc; // dense group accumulators, nval + 1 words each
    unsigned long long* kacc; // key-first entries (direct-mapped tables), nullptr: off
    unsigned long long* acc;  // [0] joined, [1] sum, [2] passing fact rows, [3] finished blocks (zeroed)
    int64_t* d_num_joined;
    int64_t* d_sum;
    int64_t* d_num_rows;
};

// x <- the lane's four rows of the step that starts at row r0 (all in the table).
__device__ __forceinline__ void pa_load4(const unsigned char* p, int type, long long r0, int lane, int64_t (&x)[4]) {
    const long long r = r0 + 2 * lane;
    if (type == TQP_I64) {
        const longlong2 a = __ldcs(reinterpret_cast<const longlong2*>(p + r * 8));
        const longlong2 b = __ldcs(reinterpret_cast<const longlong2*>(p + (r + 64) * 8));
        x[0] = a.x;
        x[1] = a.y;
        x[2] = b.x;
        x[3] = b.y;
    } else if (type == TQP_I32) {
        const int2 a = __ldcs(reinterpret_cast<const int2*>(p + r * 4));
        const int2 b = __ldcs(reinterpret_cast<const int2*>(p + (r + 64) * 4));
        x[0] = a.x;
        x[1] = a.y;
        x[2] = b.x;
        x[3] = b.y;
    } else {
        const unsigned a = __ldcs(reinterpret_cast<const unsigned short*>(p + r));
        const unsigned b = __ldcs(reinterpret_cast<const unsigned short*>(p + r + 64));
        x[0] = a & 0xFFu;
        x[1] = a >> 8;
        x[2] = b & 0xFFu;
        x[3] = b >> 8;
    }
}

__device__ __forceinline__ long long pa_row(long long r0, int lane, int j) {
    return r0 + 2 * lane + (j & 1) + 64 * (j >> 1);
}

// The same for a step that may run past the table: rows outside `in` read as 0.
template <bool kFull>
__device__ __forceinline__ void pa_col(const unsigned char* p, int type, long long r0, int lane, uint32_t in,
                                       int64_t (&x)[4]) {
    if constexpr (kFull) {
        pa_load4(p, type, r0, lane, x);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = (in >> j) & 1u ? ldg_typed(p, type, pa_row(r0, lane, j)) : 0;
    }
}

template <bool kFull>
__device__ __forceinline__ void pa_factor(const PjFactor& f, long long r0, int lane, uint32_t in, int64_t (&x)[4]) {
    const uint64_t b = static_cast<uint64_t>(f.b);
    if (f.kind == kFacConst) {
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = f.b;
        return;
    }
    pa_col<kFull>(f.p, f.type, r0, lane, in, x);
    if (f.kind == kFacPlain) return;
    const uint64_t a = f.kind == kFacAdd ? 1u : static_cast<uint64_t>(f.a);  // (kFacRsub: a is -1)
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = static_cast<int64_t>(static_cast<uint64_t>(x[j]) * a + b);
}

template <bool kFull>
__device__ __forceinline__ void pa_prod(const PjFactor (&f)[2], long long r0, int lane, uint32_t in, int64_t (&x)[4]) {
    pa_factor<kFull>(f[0], r0, lane, in, x);
    if (f[1].kind == kFacConst && f[1].b == 1) return;
    int64_t y[4];
    pa_factor<kFull>(f[1], r0, lane, in, y);
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = static_cast<int64_t>(static_cast<uint64_t>(x[j]) * static_cast<uint64_t>(y[j]));
}

// Pass bits of the lane's rows (those in `in`).
template <bool kFull, class Args>
__device__ __forceinline__ uint32_t pa_conds(const Args& A, long long r0, int lane, uint32_t in) {
    uint32_t ok = in;
    for (int q = 0; q < A.ncond; ++q) {
        const PjCond& c = A.cond[q];
        int64_t x[4];
        pa_col<kFull>(c.p, c.type, r0, lane, in, x);
        uint32_t m = 0;
        if (c.type == TQP_I64) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                m |= static_cast<uint32_t>(static_cast<uint64_t>(x[j]) - static_cast<uint64_t>(c.lo) <= c.span) << j;
        } else {
            const uint32_t lo = static_cast<uint32_t>(c.lo), sp = static_cast<uint32_t>(c.span);
#pragma unroll
            for (int j = 0; j < 4; ++j) m |= static_cast<uint32_t>(static_cast<uint32_t>(x[j]) - lo <= sp) << j;
        }
        ok &= c.negate ? ~m : m;
    }
    return ok;
}

// One row per lane (e = kPaNone: none) into the W words of entry e at
// base + e * stride: 1 (the count), then x[0..W-2].  All lanes call it.
template <int W>
__device__ __forceinline__ void pa_red(unsigned long long* base, uint32_t stride, uint32_t e,
                                       const unsigned long long (&x)[3], int lane) {
    if constexpr (W == 1) {
        if (e != kPaNone) red_add_u64(base + static_cast<unsigned long long>(e) * stride, 1ULL);
    } else {
        constexpr int P = W == 2 ? 2 : 4;  // lanes per row
        const int word = lane % P;
#pragma unroll
        for (int h = 0; h < P; ++h) {
            const int src = h * (kWarp / P) + lane / P;
            const uint32_t ee = __shfl_sync(0xffffffffu, e, src);
            unsigned long long v = 1;
#pragma unroll
            for (int i = 0; i + 1 < W; ++i) {
                const unsigned long long y = __shfl_sync(0xffffffffu, x[i], src);
                if (word == i + 1) v = y;
            }
            if (ee != kPaNone && word < W)
                red_add_u64(base + static_cast<unsigned long long>(ee) * stride + word, v);
        }
    }
}

// The step's rows of a hot entry, summed over the warp and added once. `hot` is
// the entry last seen in several lanes of a step's first row; an entry that more
// lanes hold takes its place. Absorbed rows are set to kPaNone. All lanes call it.
template <int W>
__device__ __forceinline__ void pa_combine(unsigned long long* base, uint32_t stride, uint32_t (&e)[4],
                                           const int64_t (&x0)[4], const int64_t (&x1)[4], const int64_t (&x2)[4],
                                           int lane, uint32_t& hot) {
    const uint32_t c = __shfl_sync(0xffffffffu, e[0], 0);
    const int m = c == kPaNone ? 0 : __popc(__ballot_sync(0xffffffffu, e[0] == c));
    int h = hot == kPaNone ? 0 : __popc(__ballot_sync(0xffffffffu, e[0] == hot));
    if (m > 1 && m > h) {
        hot = c;
        h = m;
    }
    if (h < 2) return;
    unsigned long long t[W] = {};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (e[j] != hot) continue;
        t[0] += 1;
        if (W > 1) t[W > 1 ? 1 : 0] += static_cast<unsigned long long>(x0[j]);
        if (W > 2) t[W > 2 ? 2 : 0] += static_cast<unsigned long long>(x1[j]);
        if (W > 3) t[W > 3 ? 3 : 0] += static_cast<unsigned long long>(x2[j]);
        e[j] = kPaNone;
    }
#pragma unroll
    for (int a = 0; a < W; ++a) {
        const unsigned long long s = static_cast<unsigned long long>(group_sum_i64(0xffffffffu, static_cast<long long>(t[a])));
        if (lane == 0) red_add_u64(base + static_cast<unsigned long long>(hot) * stride + a, s);
    }
}

// x added to entry e of a CTA's table of D entries: D counts, then per value D
// low and D high words (the low word's atomic returns what the carry needs).
// True when the 32-bit count wrapped: the CTA's own rows (below 2^31) cannot,
// the joined rows of keys with many build rows can.
__device__ __forceinline__ bool pa_smem_add(uint32_t* tab, uint32_t D, uint32_t e, int nv,
                                            const unsigned long long (&x)[3]) {
    const uint32_t c = atomicAdd(&tab[e], 1u);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a >= nv) break;
        uint32_t* lo = tab + (1 + 2 * a) * D + e;
        const uint32_t xl = static_cast<uint32_t>(x[a]);
        const uint32_t old = atomicAdd(lo, xl);
        const uint32_t xh = static_cast<uint32_t>(x[a] >> 32) + (old + xl < old ? 1u : 0u);
        if (xh) atomicAdd(lo + D, xh);
    }
    return c == ~0u;
}

// The table into global entries of nv + 1 words (neighbouring words on neighbouring lanes).
__device__ __forceinline__ void pa_smem_flush(const uint32_t* tab, uint32_t D, int nv, unsigned long long* base,
                                              uint32_t stride) {
    const uint32_t W = nv + 1;
    for (uint32_t i = threadIdx.x; i < D * W; i += blockDim.x) {
        const uint32_t e = i / W, a = i % W;
        unsigned long long x = tab[e];
        if (a > 0) {  // (also of an entry whose count wrapped to 0)
            const uint32_t* lo = tab + (2 * a - 1) * D + e;
            x = static_cast<unsigned long long>(lo[0]) | (static_cast<unsigned long long>(lo[D]) << 32);
        }
        if (x) red_add_u64(base + static_cast<unsigned long long>(e) * stride + a, x);
    }
}

// A joined row of a key with several build rows: added to each of their groups.
static __device__ __noinline__ void pa_add_chain(const ProbeAggArgs& A, uint32_t* tab, uint32_t D, uint32_t d,
                                                 uint32_t cnt, unsigned long long x0, unsigned long long x1) {
    for (uint32_t k = 0; k < cnt; ++k) {
        if (tab) {
            const unsigned long long x[3] = {x0, x1, 0};
            const uint32_t g = __ldg(&A.dgs[d]);
            if (pa_smem_add(tab, D, g, A.nval, x))  // the count's carry
                red_add_u64(A.gacc + static_cast<long long>(g) * (A.nval + 1), 1ULL << 32);
            if (k + 1 < cnt) d = __ldg(&A.next[d]);
            continue;
        }
        unsigned long long* a = A.gacc + static_cast<long long>(__ldg(&A.dgs[d])) * (A.nval + 1);
        red_add_u64(&a[0], 1ULL);
        if (A.nval > 0) red_add_u64(&a[1], x0);
        if (A.nval > 1) red_add_u64(&a[2], x1);
        if (k + 1 < cnt) d = __ldg(&A.next[d]);
    }
}

struct PaTotals {
    unsigned long long joined = 0, passed = 0;
    long long sum = 0;
};

// One warp step.  kKey: aggregate by join key (direct-mapped tables): W words
// per entry of A.kacc, no slot load; otherwise look the key up and add to the
// group of its build row(s), W = nval + 1 words (W = 0: no aggregation).
// kSmem: into the CTA's table `tab` of D entries.
template <bool kFull, bool kKey, bool kSmem, int W>
__device__ __forceinline__ void pa_step(const ProbeAggArgs& A, long long r0, int lane, bool direct, long long kmin,
                                        unsigned long long krange, uint32_t* tab, uint32_t D, PaTotals& T,
                                        uint32_t& hot) {
    uint32_t in = 0xFu;
    if constexpr (!kFull) {
        in = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) in |= static_cast<uint32_t>(pa_row(r0, lane, j) < A.n) << j;
    }
    int64_t key[4];
    pa_col<kFull>(A.fk.p, A.fk.type, r0, lane, in, key);
    // the first sum's columns are read with the key's: all loads in flight together
    int64_t v0[4] = {0, 0, 0, 0}, v1[4] = {0, 0, 0, 0}, vs[4] = {0, 0, 0, 0};
    if (A.nval > 0) pa_prod<kFull>(A.f[0], r0, lane, in, v0);
    if (W == 0 || W > 2) {
        if (A.nval > 1) pa_prod<kFull>(A.f[1], r0, lane, in, v1);
    }
    if (A.has_sum) pa_prod<kFull>(A.fs, r0, lane, in, vs);
    const uint32_t ok = pa_conds<kFull>(A, r0, lane, in);
    if (!__any_sync(0xffffffffu, ok)) return;
    T.passed += __popc(ok);
    if constexpr (kKey) {
        uint32_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned long long d = static_cast<uint64_t>(key[j]) - static_cast<uint64_t>(kmin);
            e[j] = ((ok >> j) & 1u) && d < krange ? static_cast<uint32_t>(d) : kPaNone;
            if (A.nval < 1) v0[j] = vs[j];  // (the ungrouped sum follows the group sums)
            if (A.nval < 2) v1[j] = vs[j];
        }
        if constexpr (!kSmem) pa_combine<W>(A.kacc, static_cast<uint32_t>(A.nk), e, v0, v1, vs, lane, hot);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned long long x[3] = {static_cast<unsigned long long>(v0[j]), static_cast<unsigned long long>(v1[j]),
                                             static_cast<unsigned long long>(vs[j])};
            if constexpr (kSmem) {
                if (e[j] != kPaNone) pa_smem_add(tab, D, e[j], W - 1, x);
            } else {
                pa_red<W>(A.kacc, static_cast<uint32_t>(A.nk), e[j], x, lane);
            }
        }
        return;
    }
    // the four home slots in flight together, then each row's probe sequence
    uint4 sl[4];
    uint32_t hh[4];
    const unsigned long long cap = static_cast<unsigned long long>(A.H.cap);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint64_t k = static_cast<uint64_t>(key[j]);
        bool act = (ok >> j) & 1u;
        unsigned long long h;
        if (direct) {
            h = k - static_cast<uint64_t>(kmin);
            act = act && h < cap;
        } else {
            h = k == ~0ULL ? cap : (mix64(k) & (cap - 1));
        }
        hh[j] = static_cast<uint32_t>(h);
        sl[j] = make_uint4(0u, 0u, 0u, 0u);
        if (act) sl[j] = __ldg(&A.H.slots[h]);
    }
    if (!direct) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint64_t k = static_cast<uint64_t>(key[j]);
            if (!((ok >> j) & 1u) || k == ~0ULL) continue;  // (the all-ones key lives in the extra slot)
            uint64_t sk = slot_key(sl[j]);
            for (long long i = 0; i < A.H.cap && sk != k && sk != ~0ULL; ++i) {
                hh[j] = (hh[j] + 1) & static_cast<uint32_t>(cap - 1);
                sl[j] = __ldg(&A.H.slots[hh[j]]);
                sk = slot_key(sl[j]);
            }
            if (sk != k) sl[j].w = 0;
        }
    }
    uint32_t e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        e[j] = kPaNone;
        const uint32_t cnt = sl[j].w;
        if (cnt) {
            T.joined += cnt;
            T.sum += vs[j] * static_cast<long long>(cnt);
            if (W > 0) {
                if (sl[j].z & kDirectGroup) e[j] = sl[j].z & ~kDirectGroup;
                else pa_add_chain(A, kSmem ? tab : nullptr, D, sl[j].z, cnt, static_cast<unsigned long long>(v0[j]),
                                  static_cast<unsigned long long>(v1[j]));
            }
        }
    }
    if constexpr (W > 0) {
        if constexpr (!kSmem) {
            __syncwarp();
            pa_combine<W>(A.gacc, W, e, v0, v1, vs, lane, hot);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned long long x[3] = {static_cast<unsigned long long>(v0[j]),
                                             static_cast<unsigned long long>(v1[j]), 0};
            if constexpr (kSmem) {
                if (e[j] != kPaNone) pa_smem_add(tab, D, e[j], W - 1, x);
            } else {
                pa_red<W>(A.gacc, static_cast<uint32_t>(W), e[j], x, lane);
            }
        }
    }
}

template <bool kKey, bool kSmem, int W>
__device__ __forceinline__ void pa_loop(const ProbeAggArgs& A, bool direct, long long kmin, unsigned long long krange,
                                        long long vb, long long vg, uint32_t* tab, uint32_t D, PaTotals& T) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const long long stride = vg * (kPaThreads / kWarp) * kPaStep;
    uint32_t hot = kPaNone;
    for (long long r0 = (vb * (kPaThreads / kWarp) + w) * kPaStep; r0 < A.n; r0 += stride) {
        if (r0 + kPaStep <= A.n) pa_step<true, kKey, kSmem, W>(A, r0, lane, direct, kmin, krange, tab, D, T, hot);
        else pa_step<false, kKey, kSmem, W>(A, r0, lane, direct, kmin, krange, tab, D, T, hot);
    }
}

template <bool kSmem>
__device__ __forceinline__ void pa_run(const ProbeAggArgs& A, bool bykey, bool direct, long long kmin,
                                       unsigned long long krange, long long vb, long long vg, uint32_t* tab, uint32_t D,
                                       PaTotals& T) {
    if (bykey) {
        switch (A.nval + 1 + (A.has_sum ? 1 : 0)) {
            case 1: pa_loop<true, kSmem, 1>(A, direct, kmin, krange, vb, vg, tab, D, T); break;
            case 2: pa_loop<true, kSmem, 2>(A, direct, kmin, krange, vb, vg, tab, D, T); break;
            case 3: pa_loop<true, kSmem, 3>(A, direct, kmin, krange, vb, vg, tab, D, T); break;
            default: pa_loop<true, kSmem, 4>(A, direct, kmin, krange, vb, vg, tab, D, T); break;
        }
    } else {
        switch (A.dgs ? A.nval + 1 : 0) {
            case 0: pa_loop<false, false, 0>(A, direct, kmin, 0, vb, vg, nullptr, 0, T); break;
            case 1: pa_loop<false, kSmem, 1>(A, direct, kmin, 0, vb, vg, tab, D, T); break;
            case 2: pa_loop<false, kSmem, 2>(A, direct, kmin, 0, vb, vg, tab, D, T); break;
            default: pa_loop<false, kSmem, 3>(A, direct, kmin, 0, vb, vg, tab, D, T); break;
        }
    }
}

// Block vb of vg working on this plan. kTab: the launch gave it a table of
// kPaSmemBytes (a plan whose entries cannot fit it leaves the memory to L1).
template <bool kTab>
__device__ __forceinline__ void probe_agg_block(const ProbeAggArgs& A, uint32_t* tab, long long vb, long long vg) {
    __shared__ unsigned long long red[3][kPaThreads / kWarp];
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    long long kmin = 0;
    const bool direct = ht_is_direct(A.H, &kmin);
    const bool bykey = direct && A.kacc != nullptr;
    const unsigned long long krange = bykey ? static_cast<unsigned long long>(__ldg(&A.H.meta[1]) - kmin) + 1 : 0;
    // the CTA's own table: it must fit, and be worth clearing and flushing
    const int nv = A.nval + (bykey && A.has_sum ? 1 : 0);
    const long long D = bykey ? static_cast<long long>(krange) : (A.dgs ? __ldg(A.d_groups) : 0);
    const bool smem = kTab && D > 0 && D * (4 + 8 * nv) <= kPaSmemBytes && A.n / vg >= 4 * D;
    PaTotals T;
    if (kTab && smem) {
        for (int i = threadIdx.x; i < D * (1 + 2 * nv); i += kPaThreads) tab[i] = 0;
        __syncthreads();
        pa_run<kTab>(A, bykey, direct, kmin, krange, vb, vg, tab, static_cast<uint32_t>(D), T);
        __syncthreads();
        pa_smem_flush(tab, static_cast<uint32_t>(D), nv, bykey ? A.kacc : A.gacc,
                      bykey ? static_cast<uint32_t>(A.nk) : static_cast<uint32_t>(nv + 1));
    } else {
        pa_run<false>(A, bykey, direct, kmin, krange, vb, vg, nullptr, 0, T);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        T.joined += __shfl_xor_sync(0xffffffffu, T.joined, o);
        T.passed += __shfl_xor_sync(0xffffffffu, T.passed, o);
        T.sum += __shfl_xor_sync(0xffffffffu, T.sum, o);
    }
    if (lane == 0) {
        red[0][w] = T.joined;
        red[1][w] = static_cast<unsigned long long>(T.sum);
        red[2][w] = T.passed;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    unsigned long long t[3] = {0, 0, 0};
    for (int i = 0; i < kPaThreads / kWarp; ++i)
        for (int k = 0; k < 3; ++k) t[k] += red[k][i];
    for (int k = 0; k < 3; ++k)
        if (t[k]) atomicAdd(&A.acc[k], t[k]);
    __threadfence();
    if (atomicAdd(&A.acc[3], 1ULL) != static_cast<unsigned long long>(vg) - 1ULL) return;
    __threadfence();
    // (by key: the fold writes the joined rows and the sum)
    if (A.d_num_joined && !bykey) *A.d_num_joined = static_cast<int64_t>(atomicAdd(&A.acc[0], 0ULL));
    if (A.d_sum && !bykey) *A.d_sum = static_cast<int64_t>(atomicAdd(&A.acc[1], 0ULL));
    if (A.d_num_rows) *A.d_num_rows = static_cast<int64_t>(atomicAdd(&A.acc[2], 0ULL));
}

// Host: whether the launch should give the plan a table of its own, from what
// is known before the key range and the groups are: their upper bounds.
inline bool probe_agg_tab(const ProbeAggArgs& A, long long max_groups, long long build_rows) {
    const int per = 4 + 8 * (A.nval + (A.has_sum ? 1 : 0));
    return A.dgs && (max_groups * (4 + 8 * A.nval) <= kPaSmemBytes || (A.kacc && build_rows * per <= kPaSmemBytes));
}

// Host (partjoin.cu): lower the staged probe's arguments (closed forms over
// staged columns) to the plain-load form; false when the plan falls outside
// its shapes.
struct PlanJoinArgs;
bool lower_probe_agg(const PlanJoinArgs& J, const tqp_table* F, ProbeAggArgs* A);

}  // namespace tqp
