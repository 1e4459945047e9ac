// Pair-output join in one pass over the probe keys (paper Sections 5.2-5.3;
// pairs in canonical (probe ascending, build ascending) order).
//
// What bounds it is the rate of random accesses to the build side's table
// (about one 32-byte sector per cycle and SM), then the 12 bytes per row and
// pair that stream:
//   * a table that costs one sector per probe row: 4-byte entries indexed by
//     key - min when the keys' range is at most the table's capacity; else
//     buckets of four {key, value} pairs, 32 bytes, read with one load (build
//     columns of 32 or 8 bits; 64-bit ones keep 16-byte slots);
//   * a row's match stays in registers: counts are scanned in the block, a
//     decoupled look-back over tiles gives the tile's output offset, and the
//     pairs are written at once (the staged form spilled 8 bytes per row and
//     read them back);
//   * a build side of unique keys needs no sort: the inserts store the build
//     row and raise a flag at the first second row of a key, and the sort
//     into runs (ascending rows per key) takes its row count from that flag.
// A look-back step reads 128 tiles' words, four per lane: with 8192-row tiles
// the prefix then advances faster than the tiles arrive.
// Small inputs take smaller tiles (jp_rows): 1000 rows against 100K scattered
// 64-bit keys 78 -> 50 us; 200 rows with 100K build rows each (20M pairs) 183 ->
// 29 ms, since one warp wrote them all. At 600K rows four rows per lane and 16 are
// level, at 1M 16 win (48 against 54 us). Pairs past the capacity are not walked
// through: 20K rows x 1000, counted with capacity 0, 2384 -> 144 us.
//
// Measured (60M probe rows, 1.5M unique build keys; staged form -> this): keys
// scattered over int32 1651 -> 572 us, dense 935 -> 508; 6M rows with ten build
// rows per scattered key (60M pairs) 1162 -> 358 (about 800 before the lanes of a
// warp shared the pairs of its rows). Without the look-back (offsets guessed, for
// timing) the scattered case takes 490 us, without the lookups 351.
#pragma once

#include "engine.cuh"
#include "join.cuh"

namespace tqp {

constexpr int kJpThreads = 512;
constexpr int kJpMinBlocks = 2;
constexpr int kJpWarps = kJpThreads / kWarp;
constexpr int kJpRows = 16;                       // per lane; small inputs take fewer (jp_rows)
constexpr int kJpBucket = 4;
// A value: the build row of a key's only row, flagged; or the start of the
// key's run in `bidx`, its length in `rlen`.  All ones: no row.
constexpr uint32_t kJpRow = 0x80000000u;
constexpr uint32_t kJpNone = 0xFFFFFFFFu;  // (build rows are below 2^31 - 1)

struct PairTable {
    void* mem;               // entries (uint32), buckets (uint2 x 4) or slots (uint4), all ones when free
    long long cap;           // slots, a power of two (64 or more); wide: one more for the all-ones key
    const long long* meta;   // the build keys' [min, max]
    const uint32_t* bidx;    // build rows, one run per key (when some key has several)
    const uint32_t* rlen;    // run length at the run's start
    int32_t wide;            // 64-bit build keys: uint4 {key lo, key hi, value, -}
    int32_t pad;
};

__device__ __forceinline__ bool pt_direct(const PairTable& T, unsigned long long* lo, unsigned long long* range) {
    const long long a = __ldg(&T.meta[0]), b = __ldg(&T.meta[1]);
    *lo = static_cast<unsigned long long>(a);
    *range = static_cast<unsigned long long>(b) - static_cast<unsigned long long>(a) + 1;
    return b >= a && *range - 1 < static_cast<unsigned long long>(T.cap);
}

__device__ __forceinline__ uint32_t pt_home(const PairTable& T, uint32_t key) {  // first slot of the key's bucket
    return static_cast<uint32_t>(mix64(key)) & static_cast<uint32_t>(T.cap - 1) & ~(kJpBucket - 1u);
}

// Build row i: true when its key already has a row.  *slot receives its slot.
__device__ __forceinline__ bool pt_insert(const PairTable& T, bool direct, unsigned long long lo, uint64_t key, uint32_t i,
                                          unsigned long long* slot) {
    const uint32_t val = i | kJpRow;
    if (direct) {
        *slot = key - lo;
        return atomicCAS(static_cast<uint32_t*>(T.mem) + *slot, kJpNone, val) != kJpNone;
    }
    const unsigned long long mask = static_cast<unsigned long long>(T.cap - 1);
    if (T.wide) {
        uint4* slots = static_cast<uint4*>(T.mem);
        unsigned long long h = static_cast<unsigned long long>(T.cap);
        if (key != ~0ULL) {
            h = mix64(key) & mask;
            for (long long k = 0; k < T.cap; ++k, h = (h + 1) & mask) {
                const unsigned long long prev =
                    atomicCAS(reinterpret_cast<unsigned long long*>(&slots[h]), ~0ULL, static_cast<unsigned long long>(key));
                if (prev == ~0ULL || prev == key) break;
            }
        }
        *slot = h;
        return atomicCAS(&slots[h].z, kJpNone, val) != kJpNone;
    }
    const uint32_t k32 = static_cast<uint32_t>(key);
    const unsigned long long want = (static_cast<unsigned long long>(val) << 32) | k32;
    unsigned long long* slots = static_cast<unsigned long long*>(T.mem);
    unsigned long long h = pt_home(T, k32);
    for (long long k = 0; k < T.cap; ++k, h = (h + 1) & mask) {  // (at most half full: a free slot is found)
        unsigned long long cur = *reinterpret_cast<volatile unsigned long long*>(&slots[h]);
        if (cur == ~0ULL) cur = atomicCAS(&slots[h], ~0ULL, want);
        if (cur == ~0ULL) break;
        if (static_cast<uint32_t>(cur) == k32) {
            *slot = h;
            return true;
        }
    }
    *slot = h;
    return false;
}

// The value word of a slot.
__device__ __forceinline__ uint32_t* pt_value(const PairTable& T, bool direct, unsigned long long slot) {
    uint32_t* w = static_cast<uint32_t*>(T.mem);
    return direct ? w + slot : (T.wide ? w + 4 * slot + 2 : w + 2 * slot + 1);
}

struct PairArgs {
    PairTable T;
    long long n;             // probe rows
    const unsigned char* key;
    int32_t key_type;
    int32_t kind;            // tqp_join_kind
    long long ntiles;
    int32_t* out_build;
    int32_t* out_probe;
    long long capacity;
    int64_t* d_count;
    unsigned long long* ticket;  // (zeroed)
    unsigned long long* status;  // [ntiles] look-back words (zeroed)
    int* err;
    long long wait_cap;
};

struct JpBucket {
    uint32_t w[8];  // four {key, value}
};

__device__ __forceinline__ JpBucket jp_load_bucket(const uint32_t* p) {
    JpBucket b;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(b.w[0]), "=r"(b.w[1]), "=r"(b.w[2]), "=r"(b.w[3]), "=r"(b.w[4]), "=r"(b.w[5]), "=r"(b.w[6]), "=r"(b.w[7])
        : "l"(p));
    return b;
}

// `key` in bucket b: its value, or kJpNone; *more: the next bucket may hold it.
__device__ __forceinline__ uint32_t jp_match(const JpBucket& b, uint32_t key, bool* more) {
    uint32_t v = kJpNone;
#pragma unroll
    for (int s = 0; s < kJpBucket; ++s)
        if (b.w[2 * s] == key && v == kJpNone) v = b.w[2 * s + 1];  // (a free slot's value is kJpNone)
    *more = v == kJpNone && b.w[2 * kJpBucket - 1] != kJpNone;
    return v;
}

// The values of the lane's rows r0 + 32 j; kJpNone where absent or past the table.
template <class Key, int R>
__device__ __forceinline__ void jp_lookup(const PairArgs& A, bool direct, unsigned long long lo, unsigned long long range,
                                          long long r0, uint32_t (&val)[R]) {
    constexpr int kGroup = R < 4 ? R : 4;  // rows of a lane in flight together
    const Key* kp = reinterpret_cast<const Key*>(A.key);
    const uint32_t* w = static_cast<const uint32_t*>(A.T.mem);
    if (direct) {
        unsigned long long d[R];
#pragma unroll
        for (int j = 0; j < R; ++j)
            d[j] = r0 + kWarp * j < A.n ? static_cast<unsigned long long>(static_cast<int64_t>(__ldcs(kp + r0 + kWarp * j))) - lo
                                        : ~0ULL;
#pragma unroll
        for (int j = 0; j < R; ++j) val[j] = d[j] < range ? __ldg(w + d[j]) : kJpNone;
        return;
    }
    // all key loads in flight together
    uint32_t todo = 0;
    Key x[R];
#pragma unroll
    for (int j = 0; j < R; ++j) x[j] = r0 + kWarp * j < A.n ? __ldcs(kp + r0 + kWarp * j) : Key(0);
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int64_t k = static_cast<int64_t>(x[j]);
        val[j] = static_cast<uint32_t>(k);
        // (a 64-bit probe key outside int32 has no equal key of a narrow build column)
        todo |= static_cast<uint32_t>((sizeof(Key) < 8 || k == static_cast<int32_t>(k)) && r0 + kWarp * j < A.n) << j;
    }
#pragma unroll
    for (int g = 0; g < R; g += kGroup) {
        uint32_t left = (todo >> g) & ((1u << kGroup) - 1), key[kGroup], h[kGroup];
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
            key[j] = val[g + j];
            h[j] = pt_home(A.T, key[j]);
            val[g + j] = kJpNone;
        }
        for (long long k = 0; left && k < A.T.cap; ++k) {  // (a full bucket sends a row to the next one)
            JpBucket b[kGroup];
#pragma unroll
            for (int j = 0; j < kGroup; ++j)
                if ((left >> j) & 1u) b[j] = jp_load_bucket(w + 2 * static_cast<size_t>(h[j]));
#pragma unroll
            for (int j = 0; j < kGroup; ++j) {
                if (!((left >> j) & 1u)) continue;
                bool more;
                val[g + j] = jp_match(b[j], key[j], &more);
                h[j] = (h[j] + kJpBucket) & static_cast<uint32_t>(A.T.cap - 1);
                if (!more) left &= ~(1u << j);
            }
        }
    }
}

// The value of one row of a table of 64-bit build keys.
static __device__ __noinline__ uint32_t jp_lookup_wide(const PairArgs& A, long long r) {
    if (r >= A.n) return kJpNone;
    const unsigned long long mask = static_cast<unsigned long long>(A.T.cap - 1);
    const uint4* slots = static_cast<const uint4*>(A.T.mem);
    const uint64_t key = static_cast<uint64_t>(ldg_typed(A.key, A.key_type, r));
    unsigned long long h = key == ~0ULL ? static_cast<unsigned long long>(A.T.cap) : (mix64(key) & mask);
    uint4 s = __ldg(&slots[h]);
    for (long long i = 0; i < A.T.cap && slot_key(s) != key && slot_key(s) != ~0ULL; ++i) {
        h = (h + 1) & mask;
        s = __ldg(&slots[h]);
    }
    return slot_key(s) == key ? s.z : kJpNone;  // (a free slot's value is kJpNone)
}

// Exclusive prefix of `tile` (see lookback()), 128 predecessors per step. A tile
// whose wait expired publishes its prefix marked kJpBad, and so do the tiles that
// build on it; *bad is then set.
constexpr unsigned long long kJpBad = 3ULL << 62;
__device__ __forceinline__ unsigned long long jp_lookback(unsigned long long* status, long long tile, unsigned long long agg,
                                                          int lane, int* err, long long cap, bool* bad) {
    if (lane == 0) st_relaxed_u64(&status[tile], (tile == 0 ? kFlagP : kFlagA) | agg);
    if (tile == 0) return 0;
    unsigned long long excl = 0;
    long long polls = 0;
    bool gave_up = false;
    for (long long base = tile - 1; !gave_up; base -= 4 * kWarp) {
        unsigned long long x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long idx = base - 4 * lane - k;
            x[k] = idx >= 0 ? ld_relaxed_u64(&status[idx]) : kFlagP;
        }
        while (true) {
            bool pending = false;
#pragma unroll
            for (int k = 0; k < 4; ++k) pending |= (x[k] >> 62) == 0;
            if (!__any_sync(0xffffffffu, pending)) break;
            const bool stop = (++polls > cap) || read_error(err) == TQP_ERR_TIMEOUT;
            if (__any_sync(0xffffffffu, stop)) {
                gave_up = true;
                break;
            }
            if (pending) {
                __nanosleep(32);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((x[k] >> 62) == 0) x[k] = ld_relaxed_u64(&status[base - 4 * lane - k]);
            }
        }
        if (gave_up) break;
        unsigned long long sum = 0;
        bool found = false, marked = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!found) {
                sum += x[k] & kValMask;
                marked = (x[k] >> 62) == 3;
            }
            found |= (x[k] >> 62) >= 2;
        }
        const uint32_t pmask = __ballot_sync(0xffffffffu, found);
        if (pmask) *bad = __shfl_sync(0xffffffffu, marked, __ffs(pmask) - 1);
        if (pmask && lane > __ffs(pmask) - 1) sum = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        excl += sum;
        if (pmask) break;
    }
    if (gave_up && lane == 0) latch_error(err, TQP_ERR_TIMEOUT);
    *bad |= gave_up;
    if (lane == 0) st_relaxed_u64(&status[tile], (*bad ? kJpBad : kFlagP) | ((excl + agg) & kValMask));
    return excl;
}

template <int R>
static __device__ __forceinline__ void join_pairs_tile(const PairArgs& A) {
    __shared__ long long tile_sm;
    __shared__ unsigned long long wtot[kJpWarps];
    __shared__ unsigned long long excl_sm;
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    if (threadIdx.x == 0) tile_sm = static_cast<long long>(atomicAdd(A.ticket, 1ULL));  // (every earlier tile has started)
    unsigned long long lo = 0, range = 0;
    const bool direct = pt_direct(A.T, &lo, &range);
    __syncthreads();
    const long long tile = tile_sm;
    const long long r0 = tile * (kJpThreads * R) + w * (kWarp * R) + lane;
    // pairs per row: bit j of `one` for a row of one pair; rows of longer runs in `many`
    uint32_t one = 0, many = 0;
    uint32_t val[R];
    if (!direct && A.T.wide) {
#pragma unroll
        for (int j = 0; j < R; ++j) val[j] = jp_lookup_wide(A, r0 + kWarp * j);
    } else if (A.key_type == TQP_I32) {
        jp_lookup<int32_t, R>(A, direct, lo, range, r0, val);
    } else if (A.key_type == TQP_I64) {
        jp_lookup<long long, R>(A, direct, lo, range, r0, val);
    } else {
        jp_lookup<unsigned char, R>(A, direct, lo, range, r0, val);
    }
    // inner: the row's pairs; outer: also (r, -1) without a match; semi / anti: (r, -1) or none
    const bool outer = A.kind == TQP_JOIN_LEFT_OUTER, inner = A.kind == TQP_JOIN_INNER;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const bool in = r0 + kWarp * j < A.n, hit = val[j] != kJpNone;
        const bool run = (inner || outer) && !(val[j] & kJpRow);
        const bool keep = inner ? hit && !run : (outer ? !run : hit == (A.kind == TQP_JOIN_LEFT_SEMI));
        many |= static_cast<uint32_t>(in && run) << j;
        one |= static_cast<uint32_t>(in && keep) << j;
        if (!inner && !outer) val[j] = kJpNone;  // (written as -1)
    }
    const bool flat = !__any_sync(0xffffffffu, many != 0);
    unsigned long long total = 0;  // of the warp
    if (flat) {
        total = __reduce_add_sync(0xffffffffu, __popc(one));
    } else {
#pragma unroll
        for (int j = 0; j < R; ++j)
            if ((many >> j) & 1u) total += __ldg(&A.T.rlen[val[j]]);
        total += __popc(one);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    if (lane == 0) wtot[w] = total;
    __syncthreads();
    if (w == 0) {
        unsigned long long c = lane < kJpWarps ? wtot[lane] : 0ULL, incl = c;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane < kJpWarps) wtot[lane] = incl - c;
        const unsigned long long agg = __shfl_sync(0xffffffffu, incl, kWarp - 1);
        bool bad = false;
        const unsigned long long ex = jp_lookback(A.status, tile, agg, lane, A.err, A.wait_cap, &bad);
        if (lane == 0) {
            excl_sm = ex;
            if (tile == A.ntiles - 1) {
                *A.d_count = bad ? -1 : static_cast<int64_t>(ex + agg);
                if (!bad && static_cast<long long>(ex + agg) > A.capacity) latch_error(A.err, TQP_ERR_CAPACITY);
            }
        }
    }
    __syncthreads();
    unsigned long long pos = excl_sm + wtot[w];
    const unsigned long long cap = static_cast<unsigned long long>(A.capacity);
    const uint32_t lt = lanemask_lt();
    if (flat) {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const bool k = (one >> j) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffu, k);
            const unsigned long long p = pos + __popc(m & lt);
            if (k && p < cap) {
                const uint32_t x = val[j];
                __stcs(A.out_build + p, x == kJpNone ? -1 : static_cast<int32_t>(x & ~kJpRow));
                __stcs(A.out_probe + p, static_cast<int32_t>(r0 + kWarp * j));
            }
            pos += __popc(m);
        }
        return;
    }
    for (int j = 0; j < R; ++j) {
        uint32_t x = kJpNone;
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (q == j) x = val[q];
        const bool run = (many >> j) & 1u;
        const unsigned long long c = run ? __ldg(&A.T.rlen[x]) : (one >> j) & 1u;
        unsigned long long incl = c;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const unsigned long long tot = __shfl_sync(0xffffffffu, incl, kWarp - 1);
        if (pos >= cap) {
            // (no pair of these rows is written)
        } else if (tot < (1ULL << 31)) {
            const uint32_t writes = static_cast<uint32_t>(cap - pos < tot ? cap - pos : tot);
            // the lanes share the slot's pairs: pair t belongs to the first lane whose inclusive count is above t
            const uint32_t in32 = static_cast<uint32_t>(incl), ex32 = static_cast<uint32_t>(incl - c);
            for (uint32_t t0 = 0; t0 < writes; t0 += kWarp) {
                const uint32_t t = t0 + lane;
                int o = 0;
#pragma unroll
                for (int step = kWarp / 2; step > 0; step /= 2)
                    if (__shfl_sync(0xffffffffu, in32, o + step - 1) <= t) o += step;
                const uint32_t y = __shfl_sync(0xffffffffu, x, o), first = __shfl_sync(0xffffffffu, ex32, o);
                const unsigned long long p = pos + t;
                if (t < writes) {
                    __stcs(A.out_build + p, y & kJpRow ? (y == kJpNone ? -1 : static_cast<int32_t>(y & ~kJpRow))
                                                       : static_cast<int32_t>(__ldg(&A.T.bidx[y + (t - first)])));
                    __stcs(A.out_probe + p, static_cast<int32_t>(r0 - lane + kWarp * j + o));
                }
            }
        } else {
            unsigned long long p = pos + incl - c;
            for (unsigned long long k = 0; k < c && p < cap; ++k, ++p) {
                A.out_build[p] = run ? static_cast<int32_t>(__ldg(&A.T.bidx[x + k]))
                                     : (x == kJpNone ? -1 : static_cast<int32_t>(x & ~kJpRow));
                A.out_probe[p] = static_cast<int32_t>(r0 + kWarp * j);
            }
        }
        pos += tot;
    }
}

// Rows per lane: a tile is a block's, so an input of few rows takes fewer of
// them, to spread over the SMs (and its rows over the warps that write the
// pairs of long runs).
inline int jp_rows(long long n, long long sms) {
    const long long one = kJpMinBlocks * sms * kJpThreads;  // rows that fill the chip at one per lane
    return n <= one ? 1 : (n <= 4 * one ? 4 : kJpRows);
}

}  // namespace tqp
