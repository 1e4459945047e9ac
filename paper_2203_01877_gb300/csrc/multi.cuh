// Shared scans: one pass over a table evaluates the filters of up to 32
// queries at once (each query: a conjunction of range predicates, a count of
// its passing rows and optionally the sum of a closed-form expression over
// them, exactly what tqp_filter computes without row ids).
//
// The paper runs one query at a time (Section 4.3); a served workload of many
// filter queries over one resident table would read the table once per
// query.  Here the staged scan engine streams the table once and every row is
// tested against all queries:
//   * predicates, per column: the breakpoints of every query's range
//     conditions on that column cut the value line into elementary intervals
//     on which each condition's outcome is constant; the host tabulates, per
//     interval, the 32-bit mask of queries whose conditions on that column all
//     pass.  A row's pass mask is the AND over the condition columns of the
//     mask of the interval its value falls in: a direct table lookup when the
//     breakpoints span at most kMqDirectMax values, else a branch-free binary
//     search over the sorted breakpoints.  The cost per row grows with the
//     number of condition columns, not with the number of queries;
//   * accumulation, many queries: lane q keeps query q's count and sum in
//     registers. Rows that pass some query join a queue of their warp (pass mask
//     and row, in shared memory); 32 at a time their values are computed, one row
//     per lane, and the masks are transposed (five exchange steps), so that lane q
//     holds the rows that pass query q: its count is a bit count, and it adds their
//     values;
//   * accumulation, few queries (up to kMqFew; kMqFewCounts without sums): each
//     lane keeps its own rows' totals of every query in registers. A step with more
//     than kMqQueued passing rows adds each lane's rows at once, the rest goes
//     through the queue, so that the adds of 32 rows share their instructions;
//     20M rows of four int32 columns, us, with a shared-memory atomic per (row,
//     passing query) pair / the transposed queue for any number of queries / this:
//     3 queries of 2% each 114 / 103 / 90, of 20% 193 / 258 / 114; 5 of 20% 295 /
//     291 / 137; 8 of 2% 147 / 129 / 114, of 20% 462 / 299 / 154, of 80% 566 / 559 /
//     176; 12 of 20% 657 / 314 / 293; 32 of 2% 212 / 209 / 188. Eight counts without
//     sums over two columns: 99 transposed, 118 per row.
//     The queues' shared memory is kept small because a launch shape has to fit
//     beside it: with 160 rows per warp twelve queries over six int64 columns lose a
//     resident CTA (519 -> 919 us). Few queries do without the queue where it alone
//     would cost one: every step adds its lanes' rows (10M rows of six
//     int64 columns, four queries, us: 281 with one CTA per SM, 177 so);
//   * per-query row ranges: a query may cover only rows [rlo, rhi) of the
//     scan (queries over slices of one table).  Per tile a ballot splits the
//     queries into those covering the whole tile and those touching part of
//     it; only the latter are tested row by row.
// At most two distinct sum expressions per launch (each a product of two
// affine factors of staged columns, the ProdForm of the single-query scan);
// the host splits larger query sets into groups, one launch each.
#pragma once

#include <vector>

#include "bodies.cuh"

namespace tqp {

constexpr int kMqMax = 32;          // queries per launch: one per lane
constexpr int kMqExprs = 2;         // distinct sum expressions per launch
constexpr int kMqMinPack = 3;       // smaller packs run through the single-query scan (faster there)
constexpr int kMqWords = 5120;      // mask words of all lookup tables (shared memory)
constexpr int kMqBreaks = 512;      // breakpoints of the searched tables (shared memory)
constexpr int kMqDirectMax = 4096;  // direct tables: at most this many entries per column
constexpr int kMqRows = 4;          // rows per lane of a step
constexpr int kMqFew = 8;           // launches of at most this many queries keep their totals per row, in registers

// Count-only launches: a transposed mask's bit count costs less than their rows' adds from here on.
constexpr int kMqFewCounts = 4;
inline bool mq_few(size_t nq, size_t nexpr) { return nq <= static_cast<size_t>(nexpr ? kMqFew : kMqFewCounts); }

// Queued rows (pass mask and tile row) of a consumer warp: fewer than kWarp, then
// half a step's (few queries: a whole step's where it has no more).
constexpr int kMqQueue = (1 + kMqRows / 2) * kWarp;

// Few queries: steps with at most this many passing rows use the queue. It is
// half a step because the adds of 64 queued rows cost about as much as those of a
// lane's own four; the worst sizes are those just above it, whose steps take
// either way. 20M rows of int32, one sum, us, with the line at 32 / 48 / 64 rows
// (and transposed masks for any number of queries): 8 queries that pass 25% of the
// rows 129 / 90 / 90 (111), 35% 120 / 118 / 100 (131), 45% 120 / 123 / 116 (159);
// 3 queries 25% 104 / 81 / 81 (129), 45% 90 / 92 / 100 (192).
constexpr int kMqQueued = kMqRows / 2 * kWarp;

// The queues (none where `queued` is 0: few queries only); many queries: and 32
// values of a second expression per warp (the first one's take the place of the
// rows they belong to).
__host__ __device__ constexpr int mq_queue_bytes(bool few, int nexpr, int queued) {
    return queued ? kConsumerWarps * (kMqQueue + (!few && nexpr > 1 ? kWarp : 0)) * 8 : 0;
}
// Shared memory of the queues that a launch shape has to leave room for.
constexpr int kMqShapeBytes = 3072;

// Shared memory of one launch's body: row queues | mask words | breakpoints.
__host__ __device__ constexpr int mq_words_bytes(int nwords) { return (nwords * 4 + 15) / 16 * 16; }
__host__ __device__ constexpr int mq_body_bytes(bool few, int nexpr, int queued, int nwords, int nbreaks) {
    return (mq_queue_bytes(few, nexpr, queued) + mq_words_bytes(nwords) + nbreaks * 8 + 127) / 128 * 128;
}

// One condition column of a launch.
struct MqCol {
    int32_t col;     // table column
    int32_t soff;    // byte offset of the column inside a stage
    int32_t type;
    int32_t direct;  // 1: direct table, 0: searched breakpoints
    int64_t base;    // direct: the value of entry 1 (entry 0: every smaller value)
    int32_t len;     // direct: entries (the last one: its value and every larger value);
                     // searched: breakpoints (len + 1 masks)
    int32_t off;     // first mask word
    int32_t boff;    // searched: first breakpoint
    int32_t steps;   // searched: the largest power of two <= len (0 when len == 0)
};

// Outputs and row range of one query (device memory; read at the end of the
// launch and once per chunk).
struct MqOut {
    int64_t* count;   // passing rows (nullable)
    int64_t* count2;  // a second copy of the count (nullable)
    int64_t* sum;     // sum of the query's expression (nullable)
    int64_t rlo, rhi; // rows [rlo, rhi) of the scanned table
};

struct MultiArgs {
    ScanGeom G;
    EngineCtl ctl;
    int32_t nq;
    int32_t ncols;        // condition columns
    int32_t nexpr;        // distinct sum expressions (0..kMqExprs)
    uint32_t esel;        // bit q: query q sums expression 1 (else expression 0)
    uint32_t all;         // bits of the nq queries
    int32_t nwords;       // mask words used
    int32_t nbreaks;      // breakpoints used
    int32_t body_bytes;   // shared memory of the body (mq_body_bytes, or the largest in a batch)
    int32_t queued;       // kMqQueued; 0 (few queries only): no queues
    MqCol c[kMaxStaged];
    ProdForm e[kMqExprs];
    int32_t ecol[kMqExprs][2];   // table column of each factor (-1: constant)
    const uint32_t* words;       // lookup masks (device)
    const int64_t* breaks;       // sorted breakpoints of searched tables (device)
    const MqOut* out;            // nq entries (device)
    unsigned long long* acc;     // [2 q] sum, [2 q + 1] count, [2 kMqMax] completions (zeroed)
};

// Mask of the interval containing x in column table `mc`.
__device__ __forceinline__ uint32_t mq_lookup(const MqCol& mc, int64_t x, const uint32_t* w, const int64_t* bk) {
    if (mc.direct) {
        int idx;
        if (x < mc.base) {
            idx = 0;
        } else {
            const uint64_t d = static_cast<uint64_t>(x) - static_cast<uint64_t>(mc.base);
            idx = d >= static_cast<uint64_t>(mc.len - 1) ? mc.len - 1 : static_cast<int>(d) + 1;
        }
        return w[mc.off + idx];
    }
    // number of breakpoints <= x, by halving steps over the sorted breakpoints
    const int64_t* b = bk + mc.boff;
    int pos = 0;
    for (int s = mc.steps; s > 0; s >>= 1)
        if (pos + s <= mc.len && b[pos + s - 1] <= x) pos += s;
    return w[mc.off + pos];
}

// Value of one affine factor at tile row r of a tile that is not full.
__device__ __forceinline__ int64_t mq_factor_row(const ScanGeom& G, const TileView& v, const ProdForm& f, int i,
                                                 int col, int r) {
    const int kind = f.kind[i];
    if (kind == kFacConst) return f.b[i];
    const uint64_t x = static_cast<uint64_t>(col_val(G, v, col, r));
    const uint64_t a = static_cast<uint64_t>(f.a[i]), b = static_cast<uint64_t>(f.b[i]);
    if (kind == kFacPlain) return static_cast<int64_t>(x);
    if (kind == kFacAdd) return static_cast<int64_t>(x + b);
    if (kind == kFacRsub) return static_cast<int64_t>(b - x);
    return static_cast<int64_t>(x * a + b);
}

// The transpose of the 32 x 32 bit matrix whose row l is lane l's x (all lanes
// call it): bit r of lane q's result is bit q of lane r's x.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
    uint32_t m = 0x0000FFFFu;  // columns whose index has bit j clear
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        const bool up = lane & j;
        const uint32_t keep = up ? ~m : m;
        x = (x & keep) | (__funnelshift_l(y, y, up ? 32 - j : j) & ~keep);
        m ^= m << (j >> 1);
    }
    return x;
}

// A direct-table condition column held in registers by the fast path: the
// value is clamped to [lo, lo + span] and indexes the table at word off.
struct MqHot {
    uint32_t d;     // stage byte offset | type << 20
    int32_t off;    // first mask word
    int32_t span;   // entries - 1
    int64_t lo;     // the value of entry 0's upper end (base - 1)
};
constexpr int kMqFastCols = 4;  // condition columns of the fast path

template <bool kFew>
struct MultiBody {
    static constexpr int kMinBlocks = 2;
    static constexpr int kSmemBytes = mq_body_bytes(kFew, kMqExprs, kMqQueued, kMqWords, kMqBreaks);  // the largest launch
    static constexpr int kU = kMqRows;  // rows per lane per step

    const MultiArgs& A;
    const uint32_t* w;         // shared-memory copy of the masks
    const int64_t* bk;         // shared-memory copy of the breakpoints
    unsigned long long* queue; // this warp's queued rows (pass mask, tile row << 32), and a second expression's values
    unsigned long long* val1;
    int qn = 0;                // queued rows (warp-uniform)
    unsigned long long qsum = 0;  // lane q: query q's sum and count since the last chunk
    unsigned int qcnt = 0;
    unsigned long long fsum[kMqFew] = {};  // (few queries) this lane's rows' share of them
    unsigned int fcnt[kMqFew] = {};
    int64_t rlo = 0, rhi = 0;  // lane q: query q's row range
    MqHot hot[kMqFastCols];    // fast path: the condition columns
    bool fast = false;         // every condition column has a direct table (at most kMqFastCols)

    const MqOut* outp;         // the queries' outputs and row ranges

    // Every thread of the CTA copies its share of the tables; the caller
    // synchronises the CTA before the first tile.  The tables and outputs come from the argument
    // block's pointers, or from the explicit ones (kernel parameters).
    __device__ MultiBody(const MultiArgs& a, unsigned char* sm) : MultiBody(a, sm, a.words, a.breaks, a.out) {}
    __device__ MultiBody(const MultiArgs& a, unsigned char* sm, const uint32_t* words, const int64_t* breaks,
                         const MqOut* out)
        : A(a), outp(out) {
        const int qbytes = mq_queue_bytes(kFew, a.nexpr, a.queued);
        uint32_t* ws = reinterpret_cast<uint32_t*>(sm + qbytes);
        int64_t* bs = reinterpret_cast<int64_t*>(sm + qbytes + mq_words_bytes(a.nwords));
        for (int i = threadIdx.x; i < a.nwords; i += blockDim.x) ws[i] = words[i];
        for (int i = threadIdx.x; i < a.nbreaks; i += blockDim.x) bs[i] = breaks[i];
        w = ws;
        bk = bs;
        const int warp = threadIdx.x / kWarp;
        const int lane = threadIdx.x % kWarp;
        const int cw = warp < kConsumerWarps ? warp : 0;
        queue = reinterpret_cast<unsigned long long*>(sm) + cw * kMqQueue;
        val1 = reinterpret_cast<unsigned long long*>(sm) + kConsumerWarps * kMqQueue + cw * kWarp;
        if (lane < a.nq) {
            rlo = out[lane].rlo;
            rhi = out[lane].rhi;
        }
        fast = a.ncols <= kMqFastCols;
#pragma unroll
        for (int k = 0; k < kMqFastCols; ++k) {
            hot[k] = MqHot{0u, 0, 0, 0};
            if (k < a.ncols) {
                const MqCol& mc = a.c[k];
                fast = fast && mc.direct;
                hot[k] = MqHot{static_cast<uint32_t>(mc.soff) | (static_cast<uint32_t>(mc.type) << 20), mc.off,
                               mc.len - 1, mc.base - 1};
            }
        }
    }

    // Full tiles with direct tables only: descriptors in registers, each
    // lookup a clamp and one shared-memory load.  Rows rb + lane + 32 j.
    __device__ __forceinline__ void fast_step(const ScanGeom& G, const TileView& v, int rb, int lane, uint32_t full, uint32_t part) {
        constexpr int U = kU;
        const int r0 = rb + lane;
        uint32_t m[U];
#pragma unroll
        for (int j = 0; j < U; ++j) m[j] = full;
        if (part) row_ranges<U>(v, r0, part, m);
#pragma unroll
        for (int k = 0; k < kMqFastCols; ++k) {
            if (k >= A.ncols) break;
            const MqHot h = hot[k];
            const unsigned char* col = v.stage + (h.d & 0xFFFFFu);
            const int type = static_cast<int>(h.d >> 20);
            if (type == TQP_I64) {
                const int64_t hi = h.lo + h.span;
#pragma unroll
                for (int j = 0; j < U; ++j) {
                    int64_t x = reinterpret_cast<const int64_t*>(col)[r0 + kWarp * j];
                    x = x < h.lo ? h.lo : (x > hi ? hi : x);
                    m[j] &= w[h.off + static_cast<int>(x - h.lo)];
                }
            } else {
                // 32- and 8-bit columns: the clamp bounds are values of the type
                const int lo = static_cast<int>(h.lo), hi = lo + h.span;
                int x[U];
                if (type == TQP_I32) {
#pragma unroll
                    for (int j = 0; j < U; ++j) x[j] = reinterpret_cast<const int*>(col)[r0 + kWarp * j];
                } else {
#pragma unroll
                    for (int j = 0; j < U; ++j) x[j] = col[r0 + kWarp * j];
                }
#pragma unroll
                for (int j = 0; j < U; ++j) m[j] &= w[h.off + (min(max(x[j], lo), hi) - lo)];
            }
        }
        add_rows<U>(G, v, r0, m);
    }

    // Queries whose row range ends inside the tile: their bits, row by row.
    template <int U>
    __device__ __forceinline__ void row_ranges(const TileView& v, int r0, uint32_t part, uint32_t (&m)[U]) {
        uint32_t p = part;
        while (p) {
            const int q = __ffs(p) - 1;
            p &= p - 1;
            const long long lo = __shfl_sync(0xffffffffu, static_cast<long long>(rlo), q);
            const long long hi = __shfl_sync(0xffffffffu, static_cast<long long>(rhi), q);
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const long long row = v.row0 + r0 + kWarp * j;
                if (r0 + kWarp * j < v.rows && row >= lo && row < hi) m[j] |= 1u << q;
            }
        }
    }

    // Expression e at tile row r.
    __device__ __forceinline__ unsigned long long value(const ScanGeom& G, const TileView& v, int e, int r) {
        if (!v.full)
            return static_cast<unsigned long long>(mq_factor_row(G, v, A.e[e], 0, A.ecol[e][0], r)) *
                   static_cast<unsigned long long>(mq_factor_row(G, v, A.e[e], 1, A.ecol[e][1], r));
        int64_t x[1];
        prod_eval<1>(A.e[e], v.stage, r, x);
        return static_cast<unsigned long long>(x[0]);
    }

    // The same at rows r0 + 32 j.
    template <int U>
    __device__ __forceinline__ void values(const ScanGeom& G, const TileView& v, int e, int r0, int64_t (&x)[U]) {
        if (v.full) {
            prod_eval<U>(A.e[e], v.stage, r0, x);
            return;
        }
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (r0 + kWarp * j < v.rows) x[j] = static_cast<int64_t>(value(G, v, e, r0 + kWarp * j));
    }

    // (few queries) One row into the queries it passes.
    __device__ __forceinline__ void add_row(uint32_t m, unsigned long long x0, unsigned long long x1) {
#pragma unroll
        for (int q = 0; q < kMqFew; ++q) {
            if (q >= A.nq) break;
            if (!((m >> q) & 1u)) continue;
            fsum[q] += (A.esel >> q) & 1u ? x1 : x0;
            ++fcnt[q];
        }
    }

    // The last (up to kWarp) queued rows, from `first` on, into the queries they pass.
    __device__ __forceinline__ void flush(const ScanGeom& G, const TileView& v, int first, int lane) {
        __syncwarp();
        const bool in = first + lane < qn;
        const unsigned long long t = in ? queue[first + lane] : 0ULL;
        unsigned long long x0 = 0, x1 = 0;
        if (A.nexpr > 0 && in) {
            x0 = value(G, v, 0, static_cast<int>(t >> 32));
            if (A.nexpr > 1) x1 = value(G, v, 1, static_cast<int>(t >> 32));
        }
        qn = first;
        if constexpr (kFew) {
            add_row(static_cast<uint32_t>(t), x0, x1);
            __syncwarp();  // (read before the next rows take their place)
            return;
        }
        unsigned long long* val0 = queue + first;
        __syncwarp();  // (read before the values take their place)
        val0[lane] = x0;
        if (A.nexpr > 1) val1[lane] = x1;
        __syncwarp();
        uint32_t x = warp_transpose(static_cast<uint32_t>(t), lane);  // the rows of this lane's query
        qcnt += __popc(x);
        if (A.nexpr > 0) {
            const unsigned long long* val = (A.esel >> lane) & 1u ? val1 : val0;
            for (; x; x &= x - 1) qsum += val[__ffs(x) - 1];
        }
        __syncwarp();  // (read before the next rows take their place)
    }

    // The step's rows (r0 + 32 j) into the queries they pass (every lane calls it).
    template <int U>
    __device__ __forceinline__ void add_rows(const ScanGeom& G, const TileView& v, int r0, const uint32_t (&m)[U]) {
        static_assert(U == kMqRows && U % 2 == 0, "the queue holds half a step's rows");
        const int lane = static_cast<int>(threadIdx.x % kWarp);
        const uint32_t lt = lanemask_lt();
        uint32_t b[U];
        int n = 0;
#pragma unroll
        for (int j = 0; j < U; ++j) {
            b[j] = __ballot_sync(0xffffffffu, m[j] != 0);
            n += __popc(b[j]);
        }
        if (n == 0) return;
        if constexpr (kFew) {
            if (n > A.queued) {  // many passing rows: each lane its own
                int64_t x0[U], x1[U];
#pragma unroll
                for (int j = 0; j < U; ++j) x0[j] = x1[j] = 0;
                // one copy of the code: a small scan waits for its instructions (500K rows that
                // all pass, two sums, 28 us against 34 with two; 20M rows 116 against 108)
#pragma unroll 1
                for (int e = A.nexpr - 1; e >= 0; --e) {
#pragma unroll
                    for (int j = 0; j < U; ++j) x1[j] = x0[j];
                    values<U>(G, v, e, r0, x0);
                }
#pragma unroll
                for (int j = 0; j < U; ++j)
                    add_row(m[j], static_cast<unsigned long long>(x0[j]), static_cast<unsigned long long>(x1[j]));
                return;
            }
        }
#pragma unroll
        for (int h = 0; h < U; h += U / 2) {
#pragma unroll
            for (int j = h; j < h + U / 2; ++j) {
                if (m[j])
                    queue[qn + __popc(b[j] & lt)] = m[j] | (static_cast<unsigned long long>(r0 + kWarp * j) << 32);
                qn += __popc(b[j]);
            }
            if (!kFew)
                while (qn >= kWarp) flush(G, v, qn - kWarp, lane);
        }
        if (kFew)
            while (qn >= kWarp) flush(G, v, qn - kWarp, lane);
    }

    // General path (a ragged last tile, searched tables, more than
    // kMqFastCols condition columns): rows rb + lane + 32 j of the tile.
    __device__ __forceinline__ void step(const ScanGeom& G, const TileView& v, int rb, int lane, uint32_t full,
                                         uint32_t part) {
        constexpr int U = kU;
        const int r0 = rb + lane;
        uint32_t m[U];
#pragma unroll
        for (int j = 0; j < U; ++j) m[j] = (r0 + kWarp * j < v.rows) ? full : 0u;
        if (part) row_ranges<U>(v, r0, part, m);
        // predicates: the interval masks of every condition column
        for (int k = 0; k < A.ncols; ++k) {
            const MqCol& mc = A.c[k];
            int64_t x[U];
            if (v.full) {
                load_rows<U>(v.stage + mc.soff, mc.type, r0, x);
            } else {
#pragma unroll
                for (int j = 0; j < U; ++j) x[j] = (r0 + kWarp * j < v.rows) ? col_val(G, v, mc.col, r0 + kWarp * j) : 0;
            }
#pragma unroll
            for (int j = 0; j < U; ++j) m[j] &= mq_lookup(mc, x[j], w, bk);
        }
        add_rows<U>(G, v, r0, m);
    }

    __device__ void pass1(const ScanGeom& G, const TileView& v, int cw, int lane) {
        const long long t0 = v.row0, t1 = v.row0 + v.rows;
        const bool covers = rlo <= t0 && t1 <= rhi;
        const bool touches = rlo < t1 && rhi > t0;
        const uint32_t full = __ballot_sync(0xffffffffu, covers) & A.all;
        const uint32_t part = __ballot_sync(0xffffffffu, touches && !covers) & A.all;
        if (!(full | part)) return;
        const int rw = G.T / kConsumerWarps;  // a multiple of 128
        if (v.full && fast) {
            for (int r = 0; r < rw; r += kU * kWarp) fast_step(G, v, cw * rw + r, lane, full, part);
        } else {
            for (int r = 0; r < rw && cw * rw + r < v.rows; r += kU * kWarp)
                step(G, v, cw * rw + r, lane, full, part);
        }
        if (qn > 0) flush(G, v, 0, lane);  // (the tile's columns are there until the pass ends)
    }

    __device__ void chunk_end(const ScanGeom&, long long, long long, long long, int, int lane) {
        if constexpr (kFew) {
#pragma unroll
            for (int q = 0; q < kMqFew; ++q) {
                const unsigned long long s = static_cast<unsigned long long>(
                    group_sum_i64(0xffffffffu, static_cast<long long>(fsum[q])));
                const unsigned int c = __reduce_add_sync(0xffffffffu, fcnt[q]);
                if (lane == q) {
                    qsum = s;
                    qcnt = c;
                }
                fsum[q] = 0;
                fcnt[q] = 0;
            }
        }
        const unsigned long long ls = qsum;
        const unsigned long long lc = qcnt;
        qsum = 0;
        qcnt = 0;
        if (lane < A.nq) {
            if (ls) atomicAdd(&A.acc[2 * lane], ls);
            if (lc) atomicAdd(&A.acc[2 * lane + 1], lc);
        }
        __threadfence();
        __syncwarp();
        bool last = false;
        if (lane == 0) last = last_completion(&A.acc[2 * kMqMax], A.ctl.nchunks);
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last && lane < A.nq) {
            __threadfence();
            const unsigned long long ts = atomicAdd(&A.acc[2 * lane], 0ULL);
            const unsigned long long tc = atomicAdd(&A.acc[2 * lane + 1], 0ULL);
            const MqOut& o = outp[lane];
            if (o.count) *o.count = static_cast<int64_t>(tc);
            if (o.count2) *o.count2 = static_cast<int64_t>(tc);
            if (o.sum) *o.sum = static_cast<int64_t>(ts);
        }
    }

    __device__ void finish(const ScanGeom&, int, int) {}
};

}  // namespace tqp

namespace tqp {

// The argument block of a stand-alone launch: the tables and outputs travel
// as kernel parameters (no upload, nothing to synchronise with).
struct MultiLaunch {
    MultiArgs A;
    uint32_t words[kMqWords];
    int64_t breaks[kMqBreaks];
    MqOut out[kMqMax];
};
static_assert(sizeof(MultiLaunch) <= 32764, "kernel parameters are limited to 32764 bytes");

}  // namespace tqp

// ---- host side (multi.cu) ------------------------------------------------------
namespace tqp {

// One filter query of a shared scan, lowered.
struct MqQuery {
    Cond cond[TQP_MAX_PREDS];
    int ncond = 0;
    bool has_sum = false;
    bool closed = false;   // the sum expression has the closed product form
    DExpr sum{};
    MqOut out{};
    std::vector<int> cols; // condition and expression columns, ascending
    std::vector<int> ecols; // expression columns
    std::vector<std::pair<int, int64_t>> bps;  // (column, breakpoint inside the column type's range)
    std::vector<std::pair<int, std::vector<int64_t>>> ins;  // numeric IN lists: (column, sorted values)
    bool alone = false;    // LIKE or string columns: runs through the single-query scan (and its pre-pass)
};

tqp_status mq_lower_query(const tqp_table* t, const tqp_pred* preds, int32_t npreds, const tqp_expr* sum_expr,
                          MqQuery* q);
// Pack queries into launches (first fit, in order); queries that fit no
// launch (an expression without the closed form, more than 8 columns) and
// packs of fewer than kMqMinPack queries go to `singles`, for the
// single-query scan (it reads the summed columns only at passing rows, which
// wins for one or two queries).
void mq_pack(const tqp_table* t, const std::vector<MqQuery>& qs, std::vector<std::vector<int>>* groups,
             std::vector<int>* singles);
// Lower one launch: its arguments (device pointers as offsets into `blob`,
// resolved by mq_bind once the blob is in device memory), the blob itself
// (lookup tables and per-query outputs) and the launch's shared memory.
// extra_smem: shared memory before the body (staged arguments, a batch job);
// tu: NULL for the default tuning.
tqp_status mq_lower_group(const tqp_ctx* ctx, const tqp_table* t, const std::vector<MqQuery>& qs,
                          const std::vector<int>& members, const tqp_tuning* tu, int extra_smem,
                          MultiArgs* A, std::vector<unsigned char>* blob, size_t* smem, int* ctas_per_sm);
void mq_bind(MultiArgs* A, const unsigned char* d_blob);

}  // namespace tqp
