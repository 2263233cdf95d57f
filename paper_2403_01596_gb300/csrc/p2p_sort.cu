// Device-wide exclusive scan and stable LSD radix sort (plan-time building blocks
// of the leaf binning and of the work-item / packed-layout offsets).
#include "p2p_internal.cuh"

namespace p2p_detail {

namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;  // 4096 elements per block

// Exclusive block-wide scan of one int per thread; returns the block total.
__device__ __forceinline__ int block_exclusive_scan(int v, int* smem_warp, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(P2P_FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (kScanThreads / 32) ? smem_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(P2P_FULL_MASK, w, o);
            if (lane >= o) w += y;
        }
        if (lane < (kScanThreads / 32)) smem_warp[lane] = w;  // inclusive warp prefix
    }
    __syncthreads();
    int warp_off = warp > 0 ? smem_warp[warp - 1] : 0;
    total = smem_warp[kScanThreads / 32 - 1];
    __syncthreads();
    return warp_off + x - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int32_t* __restrict__ in, int64_t n,
                                                              int32_t* __restrict__ block_sums) {
    __shared__ int warp_sums[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < n) s += in[base + i];
    int total;
    block_exclusive_scan(s, warp_sums, total);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_down(const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                            int64_t n, const int32_t* __restrict__ block_off,
                                                            int32_t* __restrict__ total_dev) {
    __shared__ int warp_sums[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int v[kScanItems];
    int s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0;
        s += v[i];
    }
    int total;
    int pre = block_exclusive_scan(s, warp_sums, total);
    const int off = block_off ? block_off[blockIdx.x] : 0;
    pre += off;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < n) out[base + i] = pre;
        pre += v[i];
    }
    if (total_dev && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total_dev = off + total;
}

// Radix sort: per pass a histogram of every tile (k_radix_hist), an exclusive scan along each digit's row of tiles
// (k_radix_rows) and the scatter, which adds the digits' totals itself.  Tiles shrink with n so that a few hundred
// blocks work on small inputs as well (at 96 000 keys 24 tiles of 4 096 left most SMs idle).  Latency bound on plans of
// ordinary size; measured on one GB300 at 70 637 points: a pass 9.5 us (18 us with a three-launch scan of all
// counts and tiles of 4 096 keys ranked 256 at a time).
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxSub = 16;  // keys per thread at most

constexpr int64_t kSortSteps[2] = {1 << 18, 1 << 22};  // largest counts with 4 and with 8 keys per thread

inline int sort_sub(int64_t n) { return n <= kSortSteps[0] ? 4 : (n <= kSortSteps[1] ? 8 : kMaxSub); }
inline int64_t sort_tiles(int64_t n) {
    const int64_t tile = (int64_t)kSortThreads * sort_sub(n);
    return n > 0 ? (n + tile - 1) / tile : 1;
}

template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const K* __restrict__ keys, int64_t n, int sub, int shift,
                                                             uint32_t mask, int32_t* __restrict__ hist, int64_t tiles) {
    __shared__ int cnt[kRadix];
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) cnt[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortThreads * sub;
    for (int c = 0; c < sub; ++c) {
        const int64_t idx = base + (int64_t)c * kSortThreads + threadIdx.x;
        if (idx < n) atomicAdd(&cnt[(uint32_t)(keys[idx] >> shift) & mask], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) hist[(int64_t)d * tiles + blockIdx.x] = cnt[d];
}

// Exclusive scan of one value per thread over a block of kSortThreads; total: the block's sum.
__device__ __forceinline__ int sort_block_scan(int v, int* warp_sum, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(P2P_FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();  // an earlier scan's sums have been read
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        before += w < warp ? warp_sum[w] : 0;
        all += warp_sum[w];
    }
    total = all;
    return before + x - v;
}

// Block d: digit d's counts over the tiles become exclusive prefixes, their sum totals[d].
__global__ void __launch_bounds__(kSortThreads) k_radix_rows(int32_t* __restrict__ hist, int64_t tiles,
                                                             int32_t* __restrict__ totals) {
    __shared__ int warp_sum[kSortWarps];
    int32_t* row = hist + (int64_t)blockIdx.x * tiles;
    int run = 0;
    for (int64_t t0 = 0; t0 < tiles; t0 += kSortThreads) {
        const int64_t t = t0 + threadIdx.x;
        const int v = t < tiles ? row[t] : 0;
        int total;
        const int pre = sort_block_scan(v, warp_sum, total);
        if (t < tiles) row[t] = run + pre;
        run += total;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

// Stable scatter.  Warp w of a tile owns 32 sub consecutive keys and ranks them in order: the lanes of a round by
// their match mask, the rounds by the warp's running count of every digit; the warps' counts are scanned once.
template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(const K* __restrict__ keys_in,
                                                                const int32_t* __restrict__ vals_in,
                                                                K* __restrict__ keys_out, int32_t* __restrict__ vals_out,
                                                                int64_t n, int sub, int shift, uint32_t mask,
                                                                const int32_t* __restrict__ hist,
                                                                const int32_t* __restrict__ totals, int64_t tiles) {
    __shared__ int cnt[kSortWarps][kRadix];
    __shared__ int warp_sum[kSortWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int w = 0; w < kSortWarps; ++w) cnt[w][tid] = 0;
    int unused;
    const int base = sort_block_scan(totals[tid], warp_sum, unused) + hist[(int64_t)tid * tiles + blockIdx.x];
    __syncthreads();
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t first = (int64_t)blockIdx.x * kSortThreads * sub + (int64_t)warp * 32 * sub + lane;
    K key[kMaxSub];
    int rank[kMaxSub];
#pragma unroll
    for (int c = 0; c < kMaxSub; ++c) {
        if (c < sub) {
            const int64_t idx = first + (int64_t)c * 32;
            const bool valid = idx < n;
            key[c] = valid ? keys_in[idx] : (K)0;
            const int d = valid ? (int)((uint32_t)(key[c] >> shift) & mask) : kRadix;  // kRadix: no key
            const unsigned peers = __match_any_sync(P2P_FULL_MASK, d);
            const int before = valid ? cnt[warp][d] : 0;
            rank[c] = before + __popc(peers & lt_mask);
            __syncwarp();
            if (valid && (__ffs(peers) - 1) == lane) cnt[warp][d] = before + __popc(peers);
            __syncwarp();
        }
    }
    __syncthreads();
    int run = base;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const int c = cnt[w][tid];
        cnt[w][tid] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kMaxSub; ++c) {
        if (c < sub) {
            const int64_t idx = first + (int64_t)c * 32;
            if (idx < n) {
                const int dst = cnt[warp][(uint32_t)(key[c] >> shift) & mask] + rank[c];
                keys_out[dst] = key[c];
                vals_out[dst] = vals_in[idx];
            }
        }
    }
}

}  // namespace

size_t scan_workspace_bytes(int64_t n) {
    if (n <= kScanTile) return 0;
    int64_t nblk = (n + kScanTile - 1) / kScanTile;
    return align_up((size_t)nblk * 4, 256) * 2 + scan_workspace_bytes(nblk);
}

cudaError_t scan_exclusive_i32(const int32_t* in, int32_t* out, int64_t n, int32_t* total_dev, void* work,
                               cudaStream_t s) {
    if (n <= 0) {
        if (total_dev) return cudaMemsetAsync(total_dev, 0, sizeof(int32_t), s);
        return cudaSuccess;
    }
    int64_t nblk = (n + kScanTile - 1) / kScanTile;
    if (nblk == 1) {
        k_scan_down<<<1, kScanThreads, 0, s>>>(in, out, n, nullptr, total_dev);
        return cudaGetLastError();
    }
    char* w = static_cast<char*>(work);
    int32_t* sums = reinterpret_cast<int32_t*>(w);
    int32_t* offs = reinterpret_cast<int32_t*>(w + align_up((size_t)nblk * 4, 256));
    void* rest = w + align_up((size_t)nblk * 4, 256) * 2;
    k_scan_reduce<<<(unsigned)nblk, kScanThreads, 0, s>>>(in, n, sums);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = scan_exclusive_i32(sums, offs, nblk, nullptr, rest, s);
    if (e != cudaSuccess) return e;
    k_scan_down<<<(unsigned)nblk, kScanThreads, 0, s>>>(in, out, n, offs, total_dev);
    return cudaGetLastError();
}

// Scratch of one sort of n pairs: counts of every tile, totals of every digit.
static size_t radix_need_bytes(int64_t n) { return align_up((size_t)sort_tiles(n) * kRadix * 4, 256) + kRadix * 4; }

// A plan sizes its scratch for a bound and sorts the pairs there are, and the larger tiles past a step need less than
// the smaller ones before it (262 144 keys 256 tiles, 262 145 keys 129): the most of all counts up to n.
size_t radix_workspace_bytes(int64_t n) {
    size_t most = radix_need_bytes(n);
    for (const int64_t step : kSortSteps)
        if (n > step && radix_need_bytes(step) > most) most = radix_need_bytes(step);
    return most;
}

template <typename K>
cudaError_t radix_sort_pairs(K* keys, int32_t* vals, K* keys_alt, int32_t* vals_alt, int64_t n, int bits, void* work,
                             size_t work_bytes, cudaStream_t s, bool* result_in_alt) {
    *result_in_alt = false;
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (work_bytes < radix_need_bytes(n)) return cudaErrorInvalidValue;
    const int64_t tiles = sort_tiles(n);
    const int sub = sort_sub(n);
    int32_t* hist = static_cast<int32_t*>(work);
    int32_t* totals = reinterpret_cast<int32_t*>(static_cast<char*>(work) + align_up((size_t)tiles * kRadix * 4, 256));
    K *kin = keys, *kout = keys_alt;
    int32_t *vin = vals, *vout = vals_alt;
    const int passes = (bits + kRadixBits - 1) / kRadixBits, pass_bits = (bits + passes - 1) / passes;
    for (int shift = 0; shift < bits; shift += pass_bits) {
        const uint32_t mask = (1u << (bits - shift < pass_bits ? bits - shift : pass_bits)) - 1u;
        k_radix_hist<K><<<(unsigned)tiles, kSortThreads, 0, s>>>(kin, n, sub, shift, mask, hist, tiles);
        k_radix_rows<<<kRadix, kSortThreads, 0, s>>>(hist, tiles, totals);
        k_radix_scatter<K><<<(unsigned)tiles, kSortThreads, 0, s>>>(kin, vin, kout, vout, n, sub, shift, mask, hist, totals,
                                                                    tiles);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        K* tk = kin;
        kin = kout;
        kout = tk;
        int32_t* tv = vin;
        vin = vout;
        vout = tv;
        *result_in_alt = !*result_in_alt;
    }
    return cudaSuccess;
}

template cudaError_t radix_sort_pairs<uint64_t>(uint64_t*, int32_t*, uint64_t*, int32_t*, int64_t, int, void*, size_t,
                                                cudaStream_t, bool*);
template cudaError_t radix_sort_pairs<uint32_t>(uint32_t*, int32_t*, uint32_t*, int32_t*, int64_t, int, void*, size_t,
                                                cudaStream_t, bool*);

}  // namespace p2p_detail
