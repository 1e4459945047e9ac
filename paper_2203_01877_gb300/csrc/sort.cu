// Stable LSD radix sort of (uint64 key, uint32 value) pairs, 8-bit digits.
//
// Used where an operator needs an order the hash table does not give: the
// group-by output (keys ascending, paper Section 5.4 / Algorithm 3's sort)
// and the join's build-side runs of equal keys.  Per pass:
//   upsweep   per-tile digit histograms (shared-memory counters);
//   scan      one block per digit: exclusive scan over tiles, plus the
//             digit's base (sum of all smaller digits' totals);
//   downsweep each warp ranks its own contiguous slice with __match_any_sync
//             peers and per-warp digit bases, so equal digits keep input
//             order (stability) and stores land in ascending position order.
// The item count lives in device memory (it is usually produced by a kernel);
// buffers and launches are sized for an upper bound, the work follows the count.
#include "host.h"

namespace tqp {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / kWarp;
constexpr int kSortItems = 16;                          // per thread
constexpr int kSortTile = kSortThreads * kSortItems;    // 4096
constexpr int kSortSlice = kSortTile / kSortWarps;      // 512 per warp
constexpr int kSortScanThreads = 1024;                  // of a scan of its own
// Blocks per SM of the shared launch: four at 64 registers wait least at the
// barriers; eight at 32 registers sort more items faster (8M build rows, each
// four times: 1001 us, with four 1088; 1.5M groups in a table of 4M: 1175, with
// four 1065).
constexpr int kSortFewBlocks = 4;
constexpr int kSortManyBlocks = 8;
constexpr long long kSortGraphItems = 1LL << 19;        // items up to which a captured sort takes a launch per step
constexpr long long kSortOneLaunch = 3LL << 20;         // items up to which the passes share a launch

// Tiles of the items there are (the buffers and launches are sized for an upper bound).
__device__ __forceinline__ long long rs_tiles(long long n) { return (n + kSortTile - 1) / kSortTile; }

// A pass of a shared launch reads what an earlier one wrote from other SMs (L2
// only); a launch of its own may read through L1, which the second read of a
// tile hits.
template <bool kShared, class T>
__device__ __forceinline__ T rs_load(const T* p) {
    if constexpr (kShared) return __ldcg(p);
    else return __ldg(p);
}

// Digit counts of tiles blockIdx.x, blockIdx.x + gridDim.x, ...
template <bool kShared>
__device__ __forceinline__ void rs_upsweep(const uint64_t* keys, long long n, int shift, uint32_t* hist, long long ntiles,
                                           unsigned long long* digit_tot, uint32_t* cnt) {
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long base = tile * kSortTile;
        cnt[threadIdx.x] = 0;
        __syncthreads();
        if (base < n) {
            for (int i = 0; i < kSortItems; ++i) {
                const long long idx = base + i * kSortThreads + threadIdx.x;
                if (idx < n) atomicAdd(&cnt[(rs_load<kShared>(&keys[idx]) >> shift) & 0xFF], 1u);
            }
        }
        __syncthreads();
        const uint32_t c = cnt[threadIdx.x];
        hist[static_cast<long long>(threadIdx.x) * ntiles + tile] = c;
        if (c) atomicAdd(&digit_tot[threadIdx.x], static_cast<unsigned long long>(c));
        if constexpr (!kShared) break;  // (a block per tile)
    }
}

// Digits blockIdx.x, blockIdx.x + gridDim.x, ...: each digit's tile counts to
// output positions (all smaller digits' totals, then the tiles before).
template <bool kShared, int kThreads>
__device__ __forceinline__ void rs_scan(uint32_t* hist, long long ntiles, const unsigned long long* digit_tot,
                                        unsigned long long* wsum) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    for (int d = blockIdx.x; d < 256; d += gridDim.x) {
        unsigned long long x = static_cast<int>(threadIdx.x) < d ? rs_load<kShared>(&digit_tot[threadIdx.x]) : 0ULL;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) wsum[w] = x;
        __syncthreads();
        unsigned long long carry = 0;
        for (int i = 0; i < kThreads / kWarp; ++i) carry += wsum[i];
        uint32_t* row = hist + static_cast<long long>(d) * ntiles;
        for (long long off = 0; off < ntiles; off += kThreads) {
            const long long i = off + threadIdx.x;
            const unsigned long long v = i < ntiles ? (kShared ? __ldcg(&row[i]) : row[i]) : 0u;
            unsigned long long incl = v;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            __syncthreads();
            if (lane == kWarp - 1) wsum[w] = incl;
            __syncthreads();
            unsigned long long before = 0, total = 0;
            for (int j = 0; j < kThreads / kWarp; ++j) {
                const unsigned long long y = wsum[j];
                before += (j < w) ? y : 0ULL;
                total += y;
            }
            if (i < ntiles) row[i] = static_cast<uint32_t>(carry + before + incl - v);
            carry += total;
        }
        __syncthreads();
    }
}

// Tiles blockIdx.x, blockIdx.x + gridDim.x, ... to their places.
template <bool kShared>
__device__ __forceinline__ void rs_downsweep(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                                             long long n, int shift, const uint32_t* hist, long long ntiles,
                                             uint32_t (*wcnt)[256]) {
    const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
    const uint32_t lt = lanemask_lt();
    for (long long tile = blockIdx.x; tile * kSortTile < n; tile += gridDim.x) {
        const long long base = tile * kSortTile;
        for (int d = lane; d < 256; d += kWarp) wcnt[w][d] = 0;
        __syncwarp();
        const long long s0 = base + static_cast<long long>(w) * kSortSlice;
        // phase 1: per-warp digit counts of the warp's slice
        for (int i = 0; i < kSortSlice / kWarp; ++i) {
            const long long idx = s0 + i * kWarp + lane;
            const int dg = idx < n ? static_cast<int>((rs_load<kShared>(&kin[idx]) >> shift) & 0xFF) : 256;
            const uint32_t peers = __match_any_sync(0xffffffffu, dg);
            if (dg < 256 && lane == __ffs(peers) - 1) wcnt[w][dg] += __popc(peers);
        }
        __syncthreads();
        // phase 2: per-warp bases = global tile offset + counts of earlier warps
        {
            const int d = threadIdx.x;  // 256 threads, one digit each
            uint32_t run = rs_load<kShared>(&hist[static_cast<long long>(d) * ntiles + tile]);
            for (int ww = 0; ww < kSortWarps; ++ww) {
                const uint32_t c = wcnt[ww][d];
                wcnt[ww][d] = run;
                run += c;
            }
        }
        __syncthreads();
        // phase 3: stable scatter
        for (int i = 0; i < kSortSlice / kWarp; ++i) {
            const long long idx = s0 + i * kWarp + lane;
            uint64_t k = 0;
            uint32_t v = 0;
            int dg = 256;
            if (idx < n) {
                k = rs_load<kShared>(&kin[idx]);
                v = rs_load<kShared>(&vin[idx]);
                dg = static_cast<int>((k >> shift) & 0xFF);
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, dg);
            if (dg < 256) {
                const uint32_t pos = wcnt[w][dg] + __popc(peers & lt);
                kout[pos] = k;
                vout[pos] = v;
            }
            __syncwarp();
            if (dg < 256 && lane == __ffs(peers) - 1) wcnt[w][dg] += __popc(peers);
            __syncwarp();
        }
        if constexpr (!kShared) break;
        __syncthreads();
    }
}

// All passes in one cooperative launch. An empty input (a build side of unique
// keys) costs this one launch instead of three per pass: 12 to 16 launches of
// about 2 us each.
template <int kBlocksPerSm>
__global__ void __launch_bounds__(kSortThreads, kBlocksPerSm) k_rs_sort(uint64_t* k0, uint32_t* v0, uint64_t* k1,
                                                                            uint32_t* v1, long long* n_ptr, int begin_bit,
                                                                            int end_bit, unsigned long long* digit_tot,
                                                                            uint32_t* hist, unsigned int* bar, int* err,
                                                                            long long wait_cap) {
    __shared__ uint32_t wcnt[kSortWarps][256];
    __shared__ unsigned long long wsum[kSortWarps];
    const long long n = *n_ptr;
    if (n == 0) return;
    const long long ntiles = rs_tiles(n);
    unsigned int arrivals = 0;
    bool ok = true;
    for (int shift = begin_bit; ok && shift < end_bit; shift += 8) {
        rs_upsweep<true>(k0, n, shift, hist, ntiles, digit_tot, wcnt[0]);
        if (!(ok = grid_barrier(bar, arrivals += gridDim.x, err, wait_cap))) break;
        rs_scan<true, kSortThreads>(hist, ntiles, digit_tot, wsum);
        if (!(ok = grid_barrier(bar, arrivals += gridDim.x, err, wait_cap))) break;
        if (blockIdx.x == 0) digit_tot[threadIdx.x] = 0;  // (read by the scans only; the next barrier orders it)
        rs_downsweep<true>(k0, v0, k1, v1, n, shift, hist, ntiles, wcnt);
        ok = grid_barrier(bar, arrivals += gridDim.x, err, wait_cap);
        uint64_t* k = k0;
        k0 = k1;
        k1 = k;
        uint32_t* v = v0;
        v0 = v1;
        v1 = v;
    }
    // a sort that gave up leaves no items: what follows takes its number from here
    if (!ok && threadIdx.x == 0) *n_ptr = 0;
}

// The same by a launch per step, where the input fills the chip and is known to
// be there: a block per tile and reads through L1. Sort-based group-by, us (one
// launch / this): 1M rows 278 / 306, 2M 450 / 472, 4M 879 / 883, 8M 1924 / 1893,
// 60M rows of 64-bit keys 19060 / 18371; a join's 8M unique build rows 183 / 261.
__global__ void __launch_bounds__(kSortThreads) k_rs_upsweep(const uint64_t* keys, const long long* n_ptr, int shift,
                                                             uint32_t* hist, unsigned long long* digit_tot) {
    __shared__ uint32_t cnt[256];
    const long long n = *n_ptr;
    rs_upsweep<false>(keys, n, shift, hist, rs_tiles(n), digit_tot, cnt);
}

__global__ void __launch_bounds__(kSortScanThreads) k_rs_scan(uint32_t* hist, const long long* n_ptr,
                                                              const unsigned long long* digit_tot) {
    __shared__ unsigned long long wsum[kSortScanThreads / kWarp];
    rs_scan<false, kSortScanThreads>(hist, rs_tiles(*n_ptr), digit_tot, wsum);
}

__global__ void __launch_bounds__(kSortThreads) k_rs_downsweep(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                                                               uint32_t* vout, const long long* n_ptr, int shift,
                                                               const uint32_t* hist) {
    __shared__ uint32_t wcnt[kSortWarps][256];
    const long long n = *n_ptr;
    rs_downsweep<false>(kin, vin, kout, vout, n, shift, hist, rs_tiles(n), wcnt);
}

// Scratch needed by radix_sort_pairs for up to n_max items.
size_t radix_sort_scratch(long long n_max) {
    const long long ntiles = (n_max + kSortTile - 1) / kSortTile;
    return 256 * sizeof(unsigned long long) + static_cast<size_t>(256) * ntiles * sizeof(uint32_t) + 256;
}

// Sort bits [begin_bit, end_bit) of the keys.  Buffers (k0, v0) hold the
// input; (k1, v1) are a second buffer of the same size.  *result_in_1 tells
// which buffer holds the sorted output.  *d_n is 0 afterwards when a wait of the
// sort expired, so kernels that read the output take the count from there.
// `fill`: how far the items are known to reach n_max.
tqp_status radix_sort_pairs(const tqp_ctx* ctx, uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, long long* d_n,
                            long long n_max, int begin_bit, int end_bit, void* scratch, cudaStream_t stream,
                            bool* result_in_1, SortFill fill) {
    *result_in_1 = false;
    if (n_max <= 0 || end_bit <= begin_bit) return TQP_OK;
    long long ntiles = (n_max + kSortTile - 1) / kSortTile;
    unsigned long long* digit_tot = static_cast<unsigned long long*>(scratch);
    unsigned int* bar = reinterpret_cast<unsigned int*>(digit_tot + 256);  // (one zeroing for both)
    uint32_t* hist = reinterpret_cast<uint32_t*>(digit_tot + 256 + 16);
    // A captured launch costs less than a barrier: a graph of a MIN plan over 1000
    // rows takes 141 us with one launch, 133 with all of them; over 2M 450 and 465.
    cudaStreamCaptureStatus captured = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &captured) != cudaSuccess) {
        cudaGetLastError();
        captured = cudaStreamCaptureStatusNone;
    }
    const bool graph = captured == cudaStreamCaptureStatusActive && n_max <= kSortGraphItems;
    if (fill == kSortAll ? n_max > kSortOneLaunch || graph : fill == kSortSome && graph) {
        const unsigned blocks = static_cast<unsigned>(ntiles);
        for (int shift = begin_bit; shift < end_bit; shift += 8) {
            TQP_CUDA(cudaMemsetAsync(digit_tot, 0, 256 * sizeof(unsigned long long), stream));
            k_rs_upsweep<<<blocks, kSortThreads, 0, stream>>>(k0, d_n, shift, hist, digit_tot);
            k_rs_scan<<<256, kSortScanThreads, 0, stream>>>(hist, d_n, digit_tot);
            k_rs_downsweep<<<blocks, kSortThreads, 0, stream>>>(k0, v0, k1, v1, d_n, shift, hist);
            TQP_CUDA(cudaGetLastError());
            std::swap(k0, k1);
            std::swap(v0, v1);
            *result_in_1 = !*result_in_1;
        }
        return TQP_OK;
    }
    TQP_CUDA(cudaMemsetAsync(digit_tot, 0, 256 * sizeof(unsigned long long) + sizeof(unsigned int), stream));
    const bool few = fill != kSortRarely;
    const void* kern = few ? reinterpret_cast<const void*>(k_rs_sort<kSortFewBlocks>)
                           : reinterpret_cast<const void*>(k_rs_sort<kSortManyBlocks>);
    const int most = std::min(resident_blocks(ctx->device, kern, kSortThreads, 0),
                              few ? kSortFewBlocks : kSortManyBlocks) * ctx->num_sms;
    const int grid = static_cast<int>(std::min<long long>(most, std::max<long long>(ntiles, 32)));
    int* err = ctx->d_err;
    long long cap = ctx->wait_cap;
    void* args[] = {&k0, &v0, &k1, &v1, &d_n, &begin_bit, &end_bit, &digit_tot, &hist, &bar, &err, &cap};
    TQP_CUDA(cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(kSortThreads), args, 0,
                                         stream));
    *result_in_1 = ((end_bit - begin_bit + 7) / 8) % 2 != 0;
    return TQP_OK;
}

}  // namespace tqp
