// String columns, IN and LIKE: the pre-pass that evaluates a scan's set and
// pattern predicates (paper Section 4.1 string representation, Section 5's
// IN / LIKE expressions).
//
// A string column is an (n x m) byte array, each string right-padded with 0.
// The pre-pass evaluates every IN / LIKE / NOT LIKE predicate of one scan in
// a single launch and writes one byte per row (1: all of them hold); the scan
// itself then filters on that byte column like on any uint8 column, so the
// staged scans, the group-bys and the plans need no string code.
//   * a warp takes 32 consecutive rows; for a string column it copies the 32
//     strings (32 m contiguous bytes, 16-byte aligned) into shared memory with
//     vector loads, and each lane then reads its own string from there;
//   * LIKE: the greedy wildcard matcher (advance on a literal or `_`, remember
//     the last `%` and resume after it on a mismatch), linear in practice;
//   * IN: binary search in the sorted, deduplicated values (int64 numbers, or
//     m-byte strings compared bytewise);
//   * the values and patterns travel in the kernel parameters and are copied
//     to shared memory once per block.
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "host.h"

namespace tqp {

constexpr int kStrThreads = 256;
constexpr int kStrWarps = kStrThreads / kWarp;
constexpr int kStrMaxWidth = 255;
// LIKE program flags: the first / last segment is anchored to the string's
// start / end; the pattern has no `%` (the one segment is the whole string);
// the greedy matcher on the raw pattern instead (a segment over 32 bytes).
constexpr int kLikeStart = 1, kLikeEnd = 2, kLikeExact = 4, kLikeGreedy = 8;
constexpr int kLikeMaxSeg = 32;

struct StrPred {
    const unsigned char* col;  // column data (device)
    int32_t type;              // TQP_CHAR or a numeric type
    int32_t width;             // string width (TQP_CHAR)
    int32_t op;                // TQP_IN, TQP_LIKE or TQP_NOT_LIKE
    int32_t off;               // byte offset of the values / pattern in the blob (8-aligned)
    int32_t count;             // IN: values; LIKE: pattern bytes
    int32_t nseg;              // LIKE: segments between `%`s
    int32_t flags;             // LIKE: kLike* flags
    int32_t prog;              // LIKE: byte offset of the segment lengths, then 256 masks per segment
    int32_t pad;
};

struct StrLaunch {
    int64_t n;
    unsigned char* out;        // n bytes
    int32_t npred;
    int32_t blob_bytes;
    int32_t stage_bytes;       // per warp: 32 strings of the widest string column (16-byte multiple)
    int32_t pad;
    StrPred p[TQP_MAX_PREDS];
    alignas(16) unsigned char blob[TQP_MAX_SET_BYTES];
};
static_assert(sizeof(StrLaunch) <= 32764, "kernel parameters are limited to 32764 bytes");

// LIKE on s[0, n) with pattern p[0, m): `%` any sequence, `_` one byte.
__device__ __forceinline__ bool like_greedy(const unsigned char* s, int n, const unsigned char* p, int m) {
    int si = 0, pi = 0, star = -1, mark = 0;
    while (si < n) {
        if (pi < m && p[pi] != '%' && (p[pi] == '_' || p[pi] == s[si])) {
            ++si;
            ++pi;
        } else if (pi < m && p[pi] == '%') {
            star = pi++;
            mark = si;
        } else if (star >= 0) {
            pi = star + 1;
            si = ++mark;
        } else {
            return false;
        }
    }
    while (pi < m && p[pi] == '%') ++pi;
    return pi == m;
}

// LIKE by segments: the pattern split at its `%`s into segments (`_` a
// one-byte wildcard inside them), each with a table of 256 masks: bit j of
// mask[c] is set when byte c may stand at the segment's position j.  An
// anchored first / last segment must match at the string's start / end; the
// segments between are found leftmost-first with the Shift-And recurrence
// (D = ((D << 1) | 1) & mask[c] per string byte), and each search starts where
// the previous segment's match ended (the leftmost choice leaves the most
// room for the rest, so it finds a match whenever one exists).
__device__ __forceinline__ bool seg_at(const unsigned char* s, int p, int len, const uint32_t* mk) {
    for (int j = 0; j < len; ++j)
        if (!((mk[s[p + j]] >> j) & 1u)) return false;
    return true;
}

__device__ bool like_segments(const unsigned char* s, int n, const StrPred& q, const unsigned char* blob) {
    const int32_t* lens = reinterpret_cast<const int32_t*>(blob + q.prog);
    const uint32_t* masks = reinterpret_cast<const uint32_t*>(blob + q.prog + ((q.nseg * 4 + 15) / 16) * 16);
    if (q.flags & kLikeExact) return n == lens[0] && seg_at(s, 0, lens[0], masks);
    int pos = 0, first = 0, last = q.nseg;
    if (q.flags & kLikeStart) {
        if (lens[0] > n || !seg_at(s, 0, lens[0], masks)) return false;
        pos = lens[0];
        first = 1;
    }
    int limit = n;  // the middle segments must end by here
    if (q.flags & kLikeEnd) {
        last = q.nseg - 1;
        limit = n - lens[last];
        if (limit < pos || !seg_at(s, limit, lens[last], masks + 256 * last)) return false;
    }
    for (int k = first; k < last; ++k) {
        const uint32_t* mk = masks + 256 * k;
        const uint32_t hit = 1u << (lens[k] - 1);
        uint32_t D = 0;
        int i = pos;
        for (; i < limit; ++i) {
            D = ((D << 1) | 1u) & mk[s[i]];
            if (D & hit) break;
        }
        if (i >= limit) return false;
        pos = i + 1;
    }
    return true;
}

// Bytewise comparison of two m-byte strings.
__device__ __forceinline__ int str_cmp(const unsigned char* a, const unsigned char* b, int m) {
    for (int i = 0; i < m; ++i)
        if (a[i] != b[i]) return a[i] < b[i] ? -1 : 1;
    return 0;
}

__global__ void __launch_bounds__(kStrThreads) k_str_prepass(const __grid_constant__ StrLaunch L) {
    extern __shared__ __align__(16) unsigned char ssm[];
    unsigned char* blob = ssm;                                           // the values and patterns
    unsigned char* stage = ssm + ((L.blob_bytes + 15) / 16) * 16;        // per warp: 32 strings
    for (int i = threadIdx.x; i < L.blob_bytes; i += blockDim.x) blob[i] = L.blob[i];
    __syncthreads();
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    unsigned char* my = stage + w * L.stage_bytes;
    const long long groups = (L.n + kWarp - 1) / kWarp;
    for (long long g = static_cast<long long>(blockIdx.x) * kStrWarps + w; g < groups;
         g += static_cast<long long>(gridDim.x) * kStrWarps) {
        const long long r0 = g * kWarp, row = r0 + lane;
        const int rows = static_cast<int>(L.n - r0 < kWarp ? L.n - r0 : kWarp);
        bool pass = lane < rows;
        for (int k = 0; k < L.npred; ++k) {
            if (!__any_sync(0xffffffffu, pass)) break;
            const StrPred& q = L.p[k];
            if (q.type == TQP_CHAR) {
                const int m = q.width;
                // the group's strings: rows * m bytes from a 16-byte aligned start
                const unsigned char* src = q.col + r0 * m;
                const int bytes = rows * m;
                __syncwarp();
                for (int i = lane; i < bytes / 16; i += kWarp)
                    reinterpret_cast<uint4*>(my)[i] = __ldg(reinterpret_cast<const uint4*>(src) + i);
                for (int i = (bytes / 16) * 16 + lane; i < bytes; i += kWarp) my[i] = __ldg(src + i);
                __syncwarp();
                if (pass) {
                    const unsigned char* s = my + lane * m;
                    if (q.op == TQP_IN) {
                        const unsigned char* v = blob + q.off;
                        int lo = 0, hi = q.count;  // first value >= s
                        while (lo < hi) {
                            const int mid = (lo + hi) / 2;
                            if (str_cmp(v + mid * m, s, m) < 0) lo = mid + 1;
                            else hi = mid;
                        }
                        pass = lo < q.count && str_cmp(v + lo * m, s, m) == 0;
                    } else {
                        int n = 0;
                        if ((m & 3) == 0) {  // four bytes at a time: the first zero byte of a word
                            const uint32_t* sw = reinterpret_cast<const uint32_t*>(s);
                            n = m;
                            for (int i = 0; i < m / 4; ++i) {
                                const uint32_t x = sw[i];
                                const uint32_t z = (x - 0x01010101u) & ~x & 0x80808080u;  // lowest set bit: first zero byte
                                if (z) {
                                    n = 4 * i + (__ffs(z) - 1) / 8;
                                    break;
                                }
                            }
                        } else {
                            while (n < m && s[n]) ++n;
                        }
                        const bool hit = (q.flags & kLikeGreedy) ? like_greedy(s, n, blob + q.off, q.count)
                                                                 : like_segments(s, n, q, blob);
                        pass = q.op == TQP_LIKE ? hit : !hit;
                    }
                }
            } else if (pass) {  // IN on a numeric column
                const int64_t x = ldg_typed(q.col, q.type, row);
                const int64_t* v = reinterpret_cast<const int64_t*>(blob + q.off);
                int lo = 0, hi = q.count;
                while (lo < hi) {
                    const int mid = (lo + hi) / 2;
                    if (v[mid] < x) lo = mid + 1;
                    else hi = mid;
                }
                pass = lo < q.count && v[lo] == x;
            }
        }
        if (lane < rows) L.out[row] = pass ? 1 : 0;
    }
}

// ---- strings of at most 32 bytes: the words in registers ---------------------------
// The general form above walks a string byte by byte through shared memory and
// is bound by integer issue. Here a lane holds its string's 32-bit words; a
// segment of a LIKE pattern is a list of 4-byte (value, mask) chunks (`_`: mask
// 0), its match positions are one 32-bit mask -- the chunk compared with the
// four-byte window at every position, later chunks ANDed in at their offset; one
// or two bytes: the positions of each byte -- and the segments are placed leftmost-first with bit operations. IN compares
// whole words against each of a short list. Still bound by issue (63% of the
// slots, 333 warp instructions per 32 strings of 24 bytes before the length was
// found with one bit scan). 20M rows, `%xy%` and a price bound: 477 -> 277 us; a
// prefix 311 -> 206, a suffix 317 -> 222, eight IN values 692 -> 275. Middle
// segments of one byte, 4M rows of 24 bytes, `a%b%c%d%e%f`: byte-wise 129, with
// windows 156, byte by byte 121. Longer lists are searched by the general form,
// and patterns of more segments or wider strings matched by it.
constexpr int kSfThreads = 256;
constexpr int kSfMinBlocks = 4;
constexpr int kSfMaxWords = 8;
constexpr int kSfSegs = 8;           // LIKE segments
constexpr int kSfNumbers = 10;       // values of a numeric IN list, many rows (sf_list); of a string one: sf_values()
constexpr int kSfWords = 1024;       // program words of a launch

struct StrFastPred {
    const unsigned char* col;
    int32_t type;
    int32_t width;
    int32_t op;
    int32_t flags;             // kLike*
    int32_t count;             // LIKE: segments; IN: values
    int32_t off;               // first program word. LIKE: {length, chunks (value, mask)} per segment; IN: the values
                               // (strings padded with zero to whole words; numbers as two words)
};

struct StrFast {
    int64_t n;
    unsigned char* out;
    int32_t npred;
    int32_t nwords;
    int32_t stage_bytes;       // per warp, for widths that are not whole words
    int32_t pad;
    StrFastPred p[TQP_MAX_PREDS];
    uint32_t words[kSfWords];
};

// The string's bytes equal to c: bit p for byte p. Seven instructions per word: a
// byte of x is zero iff neither its low seven bits carry into bit 7 nor bit 7 is
// set; the four bits are gathered at the top with one multiplication.
template <int NW>
__device__ __forceinline__ uint32_t sf_equal(const uint32_t (&w)[NW], uint32_t c) {
    const uint32_t all = c * 0x01010101u;
    uint32_t E = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const uint32_t x = w[i] ^ all;
        const uint32_t z = ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x | 0x7F7F7F7Fu);
        E = (E >> 4) | ((z * 0x00204081u) & 0xF0000000u);
    }
    return E >> (32 - 4 * NW);
}

// Match positions of a segment of `len` bytes (len >= 1): bit p set when it matches at byte p.
template <int NW>
__device__ __forceinline__ uint32_t sf_find(const uint32_t (&w)[NW], const uint32_t* chunk, int len) {
    uint32_t M = ~0u;
    if (len <= 2) {  // byte by byte: a window at every position is 20 instructions per word
        const uint32_t v = chunk[0], m = chunk[1];
        if (m & 0xFFu) M = sf_equal<NW>(w, v & 0xFFu);
        if (m & 0xFF00u) M &= sf_equal<NW>(w, (v >> 8) & 0xFFu) >> 1;
        return M;
    }
    for (int c = 0; 4 * c < len && M; ++c) {
        const uint32_t v = chunk[2 * c], m = chunk[2 * c + 1];
        uint32_t hit = 0;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t x = __funnelshift_r(w[i], i + 1 < NW ? w[i + 1] : 0u, 8 * b);
                if (((x ^ v) & m) == 0) hit |= 1u << (4 * i + b);
            }
        }
        M &= hit >> (4 * c);
    }
    return M;
}

// Word i of the string (zero past its words).
template <int NW>
__device__ __forceinline__ uint32_t sf_word(const uint32_t (&w)[NW], int i) {
    uint32_t x = 0;
#pragma unroll
    for (int j = 0; j < NW; ++j)
        if (i == j) x = w[j];
    return x;
}

template <int NW>
__device__ __forceinline__ bool sf_like(const uint32_t (&w)[NW], const StrFastPred& q, const uint32_t* prog) {
    // the string's length: its first zero byte (the lowest set bit of the first word with one)
    uint32_t z0 = 0x80u;
    int n = 4 * NW;
#pragma unroll
    for (int i = NW - 1; i >= 0; --i) {
        const uint32_t z = (w[i] - 0x01010101u) & ~w[i] & 0x80808080u;
        if (z) {
            z0 = z;
            n = 4 * i;
        }
    }
    n += (__ffs(z0) - 1) / 8;
    n = n < q.width ? n : q.width;
    int pos = 0;
    for (int k = 0; k < q.count; ++k) {
        const int len = static_cast<int>(*prog);
        const uint32_t* chunk = prog + 1;
        prog += 1 + 2 * ((len + 3) / 4);
        if (len > n - pos) return false;
        if (len == 0) return n == 0;  // (only the empty pattern has an empty segment)
        if ((q.flags & kLikeExact) || (k == 0 && (q.flags & kLikeStart))) {
            if ((q.flags & kLikeExact) && n != len) return false;
            uint32_t d = 0;
#pragma unroll
            for (int i = 0; i < NW; ++i)
                if (4 * i < len) d |= (w[i] ^ chunk[2 * i]) & chunk[2 * i + 1];
            if (d) return false;
            pos = len;
            continue;
        }
        if (k == q.count - 1 && (q.flags & kLikeEnd)) {  // at n - len (>= pos) only
            const int at = n - len, i0 = at >> 2, sh = 8 * (at & 3);
            uint32_t d = 0, lo = sf_word<NW>(w, i0);
            for (int c = 0; 4 * c < len; ++c) {
                const uint32_t hi = sf_word<NW>(w, i0 + c + 1);
                d |= (__funnelshift_r(lo, hi, sh) ^ chunk[2 * c]) & chunk[2 * c + 1];
                lo = hi;
            }
            return d == 0;
        }
        // starts from which the segment ends within the string
        uint32_t M = sf_find<NW>(w, chunk, len) & (n - len >= 31 ? ~0u : (2u << (n - len)) - 1u);
        M &= ~0u << pos;
        if (!M) return false;
        pos = __ffs(M) - 1 + len;
        if (pos >= 32 && k + 1 < q.count) return false;  // nothing is left for the next segment
    }
    return true;
}

// Two groups of 32 rows per warp step, their strings' loads in flight together.
constexpr int kSfUnroll = 2;

// The words of the lane's string in group g (zero past the width and where `pass` is false).
template <int NW>
__device__ __forceinline__ void sf_load(const StrFast& L, const StrFastPred& q, long long g, int lane, bool pass,
                                        unsigned char* my, uint32_t (&w)[NW]) {
    const int m = q.width;
#pragma unroll
    for (int i = 0; i < NW; ++i) w[i] = 0;
    if ((m & 3) == 0) {
        if (!pass) return;
        const unsigned char* s = q.col + (g * kWarp + lane) * m;
        if (m == 4 * NW) {
#pragma unroll
            for (int i = 0; i + 1 < NW; i += 2) {
                const uint2 x = __ldcs(reinterpret_cast<const uint2*>(s) + i / 2);
                w[i] = x.x;
                w[i + 1] = x.y;
            }
        } else if ((m & 7) == 0) {
#pragma unroll
            for (int i = 0; i + 1 < NW; i += 2)
                if (4 * i < m) {
                    const uint2 x = __ldcs(reinterpret_cast<const uint2*>(s) + i / 2);
                    w[i] = x.x;
                    w[i + 1] = x.y;
                }
        } else {
#pragma unroll
            for (int i = 0; i < NW; ++i)
                if (4 * i < m) w[i] = __ldcs(reinterpret_cast<const uint32_t*>(s) + i);
        }
        return;
    }
    // through shared memory: the group's strings from a 16-byte boundary, each cut out of whole words
    const long long r0 = g * kWarp;
    const int bytes = static_cast<int>(L.n - r0 < kWarp ? L.n - r0 : kWarp) * m;
    const unsigned char* src = q.col + r0 * m;
    __syncwarp();
    for (int i = lane; i < bytes / 16; i += kWarp)
        reinterpret_cast<uint4*>(my)[i] = __ldcs(reinterpret_cast<const uint4*>(src) + i);
    for (int i = (bytes / 16) * 16 + lane; i < bytes; i += kWarp) my[i] = __ldg(src + i);
    __syncwarp();
    const int at = lane * m;
    const uint32_t* sw = reinterpret_cast<const uint32_t*>(my) + at / 4;
    uint32_t x = sw[0];
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        if (4 * i >= m) break;
        const uint32_t y = sw[i + 1];
        w[i] = __funnelshift_r(x, y, 8 * (at & 3));
        x = y;
        const int left = m - 4 * i;
        if (left < 4) w[i] &= (1u << (8 * left)) - 1u;
    }
}

template <int NW>
__device__ __forceinline__ bool sf_test(const uint32_t (&w)[NW], const StrFastPred& q, const uint32_t* prog) {
    if (q.op != TQP_IN) return sf_like<NW>(w, q, prog) == (q.op == TQP_LIKE);
    const int nw = (q.width + 3) / 4;
    for (int v = 0; v < q.count; ++v) {
        uint32_t d = 0;
#pragma unroll
        for (int i = 0; i < NW; ++i)
            if (i < nw) d |= w[i] ^ prog[v * nw + i];
        if (d == 0) return true;
    }
    return false;
}

template <int NW>
__global__ void __launch_bounds__(kSfThreads, kSfMinBlocks) k_str_fast(const __grid_constant__ StrFast L) {
    extern __shared__ __align__(16) unsigned char ssm[];
    uint32_t* words = reinterpret_cast<uint32_t*>(ssm);
    for (int i = threadIdx.x; i < L.nwords; i += kSfThreads) words[i] = L.words[i];
    __syncthreads();
    const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
    unsigned char* my = ssm + (L.nwords * 4 + 15) / 16 * 16 + warp * L.stage_bytes;
    const long long groups = (L.n + kWarp - 1) / kWarp;
    const long long step = static_cast<long long>(gridDim.x) * (kSfThreads / kWarp);
    for (long long g = static_cast<long long>(blockIdx.x) * (kSfThreads / kWarp) + warp; g < groups; g += kSfUnroll * step) {
        uint32_t pass = 0;
#pragma unroll
        for (int u = 0; u < kSfUnroll; ++u) pass |= static_cast<uint32_t>((g + u * step) * kWarp + lane < L.n) << u;
        for (int k = 0; k < L.npred; ++k) {
            if (!__any_sync(0xffffffffu, pass != 0)) break;
            const StrFastPred& q = L.p[k];
            const uint32_t* prog = words + q.off;
            if (q.type != TQP_CHAR) {  // IN on a numeric column
#pragma unroll
                for (int u = 0; u < kSfUnroll; ++u) {
                    if (!((pass >> u) & 1u)) continue;
                    const uint64_t x = static_cast<uint64_t>(ldg_typed(q.col, q.type, (g + u * step) * kWarp + lane));
                    bool hit = false;
                    for (int v = 0; v < q.count; ++v)
                        hit |= prog[2 * v] == static_cast<uint32_t>(x) && prog[2 * v + 1] == static_cast<uint32_t>(x >> 32);
                    if (!hit) pass &= ~(1u << u);
                }
                continue;
            }
            uint32_t w[kSfUnroll][NW];
#pragma unroll
            for (int u = 0; u < kSfUnroll; ++u)
                if (g + u * step < groups) sf_load<NW>(L, q, g + u * step, lane, (pass >> u) & 1u, my, w[u]);
#pragma unroll
            for (int u = 0; u < kSfUnroll; ++u)
                if (((pass >> u) & 1u) && !sf_test<NW>(w[u], q, prog)) pass &= ~(1u << u);
        }
#pragma unroll
        for (int u = 0; u < kSfUnroll; ++u) {
            const long long row = (g + u * step) * kWarp + lane;
            if (row < L.n) L.out[row] = (pass >> u) & 1u;
        }
    }
}

// The longest IN list that is compared value by value; a longer one is searched
// by the general form. A value costs its words, a string that goes through shared
// memory starts behind. 4M rows, general / here, us: 12 bytes, 16 values 83 / 80,
// 24 values 86 / 89; 24 bytes, 10 values 88 / 77, 16 values 92 / 97; 25 bytes, 4
// values 80 / 77, 6 values 82 / 87; int32, 10 values 56 / 56, 12 values 55 / 58.
// Few rows wait for memory and launches, not for issue, and longer lists win too: 27
// bytes, 8 values of a text (of random letters), here / general, 400K rows 0.87
// (0.84), 1M 0.94 (0.97), 2M 1.00 (1.13), 16M 1.12 (1.43); 32 values 200K 0.83
// (0.80), 400K 1.03 (1.04), 700K 1.24 (1.27).
static int sf_list(long long n, int most) {
    if (n < (1LL << 19)) return 32;
    return n < 3 * (1LL << 19) ? std::max(most, 10) : most;
}
static int sf_values(int nw, bool stage) { return stage ? std::min(14, 36 / nw) : 64 / nw; }

// The launch above from the general one; false outside its shapes.
static bool lower_str_fast(const StrLaunch& L, StrFast* F, int* words_per_string) {
    F->n = L.n;
    F->out = L.out;
    F->npred = L.npred;
    int used = 0, maxw = 4;
    bool stage = false;
    auto push = [&](uint32_t x) {
        if (used < kSfWords) F->words[used] = x;
        ++used;
    };
    for (int k = 0; k < L.npred; ++k) {
        const StrPred& q = L.p[k];
        StrFastPred& f = F->p[k];
        f = StrFastPred{q.col, q.type, q.width, q.op, q.flags, q.count, used};
        const unsigned char* data = L.blob + q.off;
        if (q.type == TQP_CHAR) {
            if (q.width > 4 * kSfMaxWords) return false;
            maxw = std::max(maxw, q.width);
            stage = stage || q.width % 4 != 0;
        }
        if (q.op == TQP_IN) {
            if (q.type != TQP_CHAR && q.count > sf_list(L.n, kSfNumbers)) return false;
            const int bytes = q.type == TQP_CHAR ? q.width : 8;
            for (int v = 0; v < q.count; ++v)
                for (int b = 0; b < bytes; b += 4) {
                    uint32_t x = 0;
                    for (int i = 0; i < 4 && b + i < bytes; ++i) x |= static_cast<uint32_t>(data[v * bytes + b + i]) << (8 * i);
                    push(x);
                }
            continue;
        }
        if ((q.flags & kLikeGreedy) || q.nseg > kSfSegs) return false;
        f.count = q.nseg;
        // the segments again, from the pattern (split at `%`; without one, the whole pattern)
        std::vector<std::string> segs;
        if (q.flags & kLikeExact) {
            segs.emplace_back(reinterpret_cast<const char*>(data), q.count);
        } else {
            std::string cur;
            for (int i = 0; i <= q.count; ++i) {
                if (i < q.count && data[i] != '%') {
                    cur.push_back(static_cast<char>(data[i]));
                } else {
                    if (!cur.empty()) segs.push_back(cur);
                    cur.clear();
                }
            }
        }
        for (const std::string& g : segs) {
            push(static_cast<uint32_t>(g.size()));
            for (size_t b = 0; b < g.size(); b += 4) {
                uint32_t x = 0, m = 0;
                for (size_t i = 0; i < 4 && b + i < g.size(); ++i) {
                    if (g[b + i] == '_') continue;
                    x |= static_cast<uint32_t>(static_cast<unsigned char>(g[b + i])) << (8 * i);
                    m |= 0xFFu << (8 * i);
                }
                push(x);
                push(m);
            }
        }
    }
    if (used > kSfWords) return false;
    F->nwords = used;
    F->stage_bytes = stage ? (kWarp * maxw + 4 + 15) / 16 * 16 : 0;
    const int nw = maxw <= 8 ? 2 : (maxw <= 16 ? 4 : (maxw <= 24 ? 6 : 8));
    *words_per_string = nw;
    for (int k = 0; k < L.npred; ++k)
        if (L.p[k].op == TQP_IN && L.p[k].type == TQP_CHAR && L.p[k].count > sf_list(L.n, sf_values(nw, stage)))
            return false;
    return true;
}

template <int NW>
static tqp_status launch_str_fast(const tqp_ctx* ctx, const StrFast& F, cudaStream_t st) {
    const size_t smem = (static_cast<size_t>(F.nwords) * 4 + 15) / 16 * 16 +
                        static_cast<size_t>(kSfThreads / kWarp) * F.stage_bytes;  // (below 16 KB)
    const long long groups = (F.n + kWarp - 1) / kWarp;
    const long long want = (groups + kSfThreads / kWarp - 1) / (kSfThreads / kWarp);
    const long long grid = std::min<long long>(want, 1LL * kSfMinBlocks * ctx->num_sms);
    k_str_fast<NW><<<static_cast<unsigned>(grid), kSfThreads, smem, st>>>(F);
    TQP_CUDA(cudaGetLastError());
    return TQP_OK;
}

static bool is_set_op(int op) { return op == TQP_IN || op == TQP_LIKE || op == TQP_NOT_LIKE; }

bool has_set_preds(const tqp_table* t, const tqp_pred* preds, int32_t npreds) {
    for (int i = 0; i < npreds && i < TQP_MAX_PREDS && preds; ++i) {
        if (is_set_op(preds[i].op)) return true;
        if (preds[i].col >= 0 && preds[i].col < t->num_cols && t->cols[preds[i].col].type == TQP_CHAR) return true;
    }
    return false;
}

tqp_status str_prepass(tqp_ctx* ctx, const tqp_table* t, const tqp_pred* preds, int32_t npreds, cudaStream_t st,
                       StrLowered* out, bool check_only) {
    out->active = false;
    out->t = *t;
    out->npreds = npreds;
    if (npreds < 0 || npreds > TQP_MAX_PREDS)
        return fail(TQP_ERR_INVALID_ARG, "npreds %d outside [0, %d]", npreds, TQP_MAX_PREDS);
    if (npreds > 0 && !preds) return fail(TQP_ERR_INVALID_ARG, "preds is NULL");
    for (int i = 0; i < npreds; ++i) out->preds[i] = preds[i];
    if (!has_set_preds(t, preds, npreds)) return TQP_OK;
    std::vector<unsigned char> lb(sizeof(StrLaunch), 0);
    StrLaunch* L = reinterpret_cast<StrLaunch*>(lb.data());
    std::vector<int> cols;
    int nkeep = 0;
    size_t used = 0;
    int maxw = 0;
    for (int i = 0; i < npreds; ++i) {
        const tqp_pred& p = preds[i];
        if (p.col < 0 || p.col >= t->num_cols)
            return fail(TQP_ERR_INVALID_ARG, "predicate %d: column %d out of range", i, p.col);
        const tqp_column& c = t->cols[p.col];
        const bool str = c.type == TQP_CHAR;
        if (!is_set_op(p.op)) {
            if (str)
                return fail(TQP_ERR_INVALID_ARG, "predicate %d: string column %d takes IN / LIKE / NOT LIKE only", i,
                            p.col);
            out->preds[nkeep++] = p;
            continue;
        }
        if (!str && p.op != TQP_IN)
            return fail(TQP_ERR_INVALID_ARG, "predicate %d: LIKE on numeric column %d", i, p.col);
        if (p.hi < 0 || (p.hi > 0 && p.lo == 0))
            return fail(TQP_ERR_INVALID_ARG, "predicate %d: bad value list (lo %lld, hi %lld)", i, (long long)p.lo,
                        (long long)p.hi);
        if (p.op != TQP_IN && p.hi > kStrMaxWidth)
            return fail(TQP_ERR_INVALID_ARG, "predicate %d: LIKE pattern longer than %d bytes", i, kStrMaxWidth);
        StrPred& q = L->p[L->npred++];
        q.col = static_cast<const unsigned char*>(c.data);
        q.type = c.type;
        q.width = str ? c.scale : 0;
        maxw = std::max(maxw, q.width);
        q.op = p.op;
        q.off = static_cast<int32_t>(used);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(static_cast<uintptr_t>(p.lo));
        std::vector<unsigned char> data;
        if (p.op != TQP_IN) {  // the pattern
            data.assign(src, src + p.hi);
            q.count = static_cast<int32_t>(p.hi);
        } else if (str) {      // m-byte strings, sorted and deduplicated
            const int m = c.scale;
            std::vector<std::string> v;
            for (long long k = 0; k < p.hi; ++k) v.emplace_back(reinterpret_cast<const char*>(src) + k * m, m);
            std::sort(v.begin(), v.end(), [](const std::string& a, const std::string& b) {
                return memcmp(a.data(), b.data(), a.size()) < 0;
            });
            v.erase(std::unique(v.begin(), v.end()), v.end());
            for (const std::string& x : v) data.insert(data.end(), x.begin(), x.end());
            q.count = static_cast<int32_t>(v.size());
        } else {               // int64 numbers, sorted and deduplicated
            std::vector<int64_t> v(reinterpret_cast<const int64_t*>(src), reinterpret_cast<const int64_t*>(src) + p.hi);
            std::sort(v.begin(), v.end());
            v.erase(std::unique(v.begin(), v.end()), v.end());
            data.resize(v.size() * 8);
            if (!v.empty()) memcpy(data.data(), v.data(), data.size());
            q.count = static_cast<int32_t>(v.size());
        }
        if (used + data.size() > static_cast<size_t>(TQP_MAX_SET_BYTES))
            return fail(TQP_ERR_UNSUPPORTED, "IN / LIKE values take more than %d bytes", TQP_MAX_SET_BYTES);
        if (!data.empty()) memcpy(L->blob + used, data.data(), data.size());
        used = (used + data.size() + 15) / 16 * 16;
        if (p.op != TQP_IN) {  // the segment program, when it fits (else the greedy matcher)
            std::vector<std::vector<unsigned char>> segs;
            std::vector<unsigned char> cur;
            bool any_pct = false;
            for (unsigned char ch : data) {
                if (ch == '%') {
                    any_pct = true;
                    if (!cur.empty()) segs.push_back(cur);
                    cur.clear();
                } else {
                    cur.push_back(ch);
                }
            }
            if (!cur.empty() || !any_pct) segs.push_back(cur);
            q.nseg = static_cast<int32_t>(segs.size());
            q.flags = any_pct ? 0 : kLikeExact;
            if (any_pct && data.front() != '%') q.flags |= kLikeStart;
            if (any_pct && data.back() != '%') q.flags |= kLikeEnd;
            bool fits = true;
            for (const auto& g : segs) fits = fits && g.size() <= static_cast<size_t>(kLikeMaxSeg);
            const size_t hdr = (segs.size() * 4 + 15) / 16 * 16;
            const size_t prog_bytes = hdr + segs.size() * 256 * 4;
            if (!fits || used + prog_bytes > static_cast<size_t>(TQP_MAX_SET_BYTES)) {
                q.flags = kLikeGreedy;
            } else {
                q.prog = static_cast<int32_t>(used);
                int32_t* lens = reinterpret_cast<int32_t*>(L->blob + used);
                uint32_t* masks = reinterpret_cast<uint32_t*>(L->blob + used + hdr);
                for (size_t k = 0; k < segs.size(); ++k) {
                    lens[k] = static_cast<int32_t>(segs[k].size());
                    for (size_t j = 0; j < segs[k].size(); ++j)
                        for (int c = 0; c < 256; ++c)
                            if (segs[k][j] == '_' || segs[k][j] == c) masks[k * 256 + c] |= 1u << j;
                }
                used += prog_bytes;
            }
        }
        cols.push_back(p.col);
    }
    TQP_TRY(check_device_cols(t, cols, "IN / LIKE"));
    if (t->num_cols + 1 > TQP_MAX_COLS)
        return fail(TQP_ERR_UNSUPPORTED, "IN / LIKE need a free column slot (the table has %d of %d)", t->num_cols,
                    TQP_MAX_COLS);
    if (check_only) {  // the other predicates, as the scan will take them; nothing allocated or launched
        out->npreds = nkeep;
        return TQP_OK;
    }
    // the pass column, then the table with it appended and the predicate on it
    const long long n = t->num_rows;
    unsigned char* pass = nullptr;
    if (n > 0) {
        pass = static_cast<unsigned char*>(arena_alloc(ctx, static_cast<size_t>((n + 15) / 16 * 16)));
        if (!pass) return arena_oom(ctx, static_cast<size_t>((n + 15) / 16 * 16));
        L->n = n;
        L->out = pass;
        L->blob_bytes = static_cast<int32_t>(used);
        StrFast F;
        int nw = 0;
        if (lower_str_fast(*L, &F, &nw)) {
            TQP_TRY(nw == 2 ? launch_str_fast<2>(ctx, F, st)
                            : (nw == 4 ? launch_str_fast<4>(ctx, F, st)
                                       : (nw == 6 ? launch_str_fast<6>(ctx, F, st) : launch_str_fast<8>(ctx, F, st))));
        } else {
            L->stage_bytes = (kWarp * maxw + 15) / 16 * 16;
            static SmemFlags attr;
            TQP_TRY(allow_smem(ctx, reinterpret_cast<const void*>(k_str_prepass), attr));
            const size_t smem = (used + 15) / 16 * 16 + static_cast<size_t>(kStrWarps) * L->stage_bytes;
            int occ = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_str_prepass, kStrThreads, smem) != cudaSuccess ||
                occ < 1)
                occ = 1;
            const long long groups = (n + kWarp - 1) / kWarp;
            const long long want = (groups + kStrWarps - 1) / kStrWarps;
            const int grid = static_cast<int>(std::min<long long>(want, static_cast<long long>(ctx->num_sms) * occ));
            k_str_prepass<<<grid, kStrThreads, smem, st>>>(*L);
            TQP_CUDA(cudaGetLastError());
        }
    }
    out->cols.assign(t->cols, t->cols + t->num_cols);
    tqp_column pc;
    pc.data = pass;
    pc.type = TQP_U8;
    pc.scale = 0;
    out->cols.push_back(pc);
    out->t.num_cols = t->num_cols + 1;
    out->t.cols = out->cols.data();
    tqp_pred eq;
    eq.col = t->num_cols;
    eq.op = TQP_EQ;
    eq.lo = 1;
    eq.hi = 0;
    out->preds[nkeep++] = eq;
    out->npreds = nkeep;
    out->active = true;
    return TQP_OK;
}

}  // namespace tqp
