// Leaf binning (Sec. 3.1, Morton order of Sec. 3.2), neighbour lists (Sec. 3.2,
// 27-box 3D neighbourhood) and plan construction including the redundant
// per-box packed layout (Sec. 3.3, eq. 6 - 8, collected on the device).
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "p2p_internal.cuh"

namespace p2p_detail {

static thread_local char g_last_error[512] = "";

void set_cuda_error(cudaError_t e, const char* where) {
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s (%s)", where, cudaGetErrorString(e), cudaGetErrorName(e));
}

void set_message(const char* msg) { snprintf(g_last_error, sizeof(g_last_error), "%s", msg); }

}  // namespace p2p_detail

using namespace p2p_detail;

// Box-group kernel tables (p2p_group.cu).
cudaError_t p2p_group_build(p2p_plan* p, const int32_t* nbr_ptr, const int32_t* nbr_idx, uint32_t* keys,
                            int32_t* vals, uint32_t* keys_alt, int32_t* vals_alt, void* radix_ws, size_t radix_bytes,
                            int32_t* maxes, cudaStream_t s, int32_t* cap);

// Tensor-core lists (p2p_tc.cu).
cudaError_t p2p_tc_build(p2p_plan* p, int32_t* bound, int32_t* units, void* scan_ws, cudaStream_t s);
cudaError_t p2p_tcb_build(p2p_plan* p, int32_t* scratch, void* scan_ws, cudaStream_t s);

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(int64_t n, int per_block) { return (unsigned)((n + per_block - 1) / per_block); }

// ------------------------------------------------------------------ binning --

// cell = clamp(floor((double(x) - lo) / h), 0, ng - 1), with explicitly rounded
// double operations so no contraction can change the result.
__device__ __forceinline__ uint32_t cell_of(float x, double lo, double h, int ng) {
    double t = __ddiv_rn(__dsub_rn((double)x, lo), h);
    double f = floor(t);
    if (f < 0.0) f = 0.0;
    if (f > (double)(ng - 1)) f = (double)(ng - 1);
    return (uint32_t)f;
}

// The same cell from FP32 arithmetic where that is safe: q = (x - lo) / h evaluated in floats is off by less than
// (4 |q| + |lo| / h + 1) 2^-23 (rounding of lo, the difference, 1 / h and the product), so a q further than that from
// every integer has the right floor; the others take the double division.  FP64 runs at 1/64 of the FP32 rate here:
// 2^20 points took 83 us in doubles.
struct AxisGrid {
    double lo, h;
    float lo_f, inv_h, slack;  // slack: (|lo| / h + 1) 2^-23
};
__device__ __forceinline__ uint32_t cell_fast(float x, const AxisGrid& g, int ng) {
    const float q = (x - g.lo_f) * g.inv_h;
    const float f = floorf(q);
    const float off = fminf(q - f, f + 1.f - q);
    if (!(off > fmaf(fabsf(q), 4.8e-7f, g.slack))) return cell_of(x, g.lo, g.h, ng);  // also where q is not finite
    return (uint32_t)fminf(fmaxf(f, 0.f), (float)(ng - 1));
}

template <typename K>
__global__ void k_keys(const float* __restrict__ pts, int64_t n, AxisGrid g0, AxisGrid g1, AxisGrid g2, int ng,
                       K* __restrict__ keys, int32_t* __restrict__ vals, int32_t* __restrict__ bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x = pts[3 * i], y = pts[3 * i + 1], z = pts[3 * i + 2];
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) {
        *bad = 1;
        x = y = z = 0.f;
    }
    keys[i] = (K)p2p_morton(cell_fast(x, g0, ng), cell_fast(y, g1, ng), cell_fast(z, g2, ng));
    vals[i] = (int32_t)i;
}

// Boxes are the runs of equal sorted keys.  A block of kThreads threads takes kHeads consecutive keys per thread:
// k_heads counts the run heads of every block, k_rle numbers them from the scanned counts and writes the boxes.
constexpr int kHeads = 4;
template <typename K>
__device__ __forceinline__ int heads_of(const K* __restrict__ keys, int64_t n, int64_t s0, bool (&head)[kHeads]) {
    K prev = s0 > 0 && s0 < n ? keys[s0 - 1] : (K)0;
    int c = 0;
#pragma unroll
    for (int i = 0; i < kHeads; ++i) {
        const bool in = s0 + i < n;
        const K k = in ? keys[s0 + i] : (K)0;
        head[i] = in && (s0 + i == 0 || k != prev);
        prev = k;
        c += head[i];
    }
    return c;
}

template <typename K>
__global__ void __launch_bounds__(kThreads) k_heads(const K* __restrict__ keys, int64_t n, int32_t* __restrict__ count) {
    const int64_t s0 = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * kHeads;
    bool head[kHeads];
    int c = heads_of(keys, n, s0, head);
    __shared__ int sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    c = __reduce_add_sync(P2P_FULL_MASK, c);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x == 0) count[blockIdx.x] = sum;
}

template <typename K>
__global__ void __launch_bounds__(kThreads)
    k_rle(const K* __restrict__ keys, const int32_t* __restrict__ vals, const int32_t* __restrict__ first, int64_t n,
          int32_t* __restrict__ perm, int32_t* __restrict__ point_box, int64_t* __restrict__ box_keys,
          int32_t* __restrict__ box_ptr) {
    __shared__ int warp_sum[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s0 = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * kHeads;
    bool head[kHeads];
    const int c = heads_of(keys, n, s0, head);
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(P2P_FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    int id = first[blockIdx.x] + x - c - 1;  // the run that position s0 - 1 belongs to
    for (int w = 0; w < warp; ++w) id += warp_sum[w];
#pragma unroll
    for (int i = 0; i < kHeads; ++i) {
        const int64_t s = s0 + i;
        if (s >= n) break;
        if (head[i]) {
            ++id;
            box_keys[id] = (int64_t)keys[s];
            box_ptr[id] = (int32_t)s;
        }
        const int32_t orig = vals[s];
        perm[s] = orig;
        point_box[orig] = id;
        if (s == n - 1) box_ptr[id + 1] = (int32_t)n;
    }
}

// --------------------------------------------------------------- neighbours --

__device__ __forceinline__ int32_t find_key(const int64_t* __restrict__ keys, int32_t nb, int64_t key) {
    int32_t lo = 0, hi = nb - 1;
    while (lo <= hi) {
        int32_t mid = lo + ((hi - lo) >> 1);
        int64_t v = __ldg(keys + mid);
        if (v == key) return mid;
        if (v < key) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// Ascending bitonic sort of one int per lane across the warp.
__device__ __forceinline__ int32_t warp_sort_asc(int32_t v, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            int32_t o = __shfl_xor_sync(P2P_FULL_MASK, v, j);
            bool up = (lane & k) == 0;
            bool lower = (lane & j) == 0;
            v = (lower == up) ? min(v, o) : max(v, o);
        }
    }
    return v;
}

// One warp per target box; lane l < 27 probes the offset (l%3-1, (l/3)%3-1, l/9-1) among the source boxes' keys (the
// same keys for a one-set structure, TWO = false) and keeps what it found; sum: the sources of all neighbourhoods.
template <bool TWO>
__global__ void __launch_bounds__(kThreads)
    k_nbr_find(const int64_t* __restrict__ box_keys, int32_t nb, const int64_t* __restrict__ src_keys, int32_t nbs,
               const int32_t* __restrict__ src_box_ptr, int ng, int32_t* __restrict__ cnt, int32_t* __restrict__ found,
               unsigned long long* __restrict__ sum, int32_t* __restrict__ bad) {
    __shared__ unsigned long long block_sum;
    if (threadIdx.x == 0) block_sum = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b < nb) {
        const uint64_t key = (uint64_t)box_keys[b];
        const int cx = (int)p2p_compact3(key), cy = (int)p2p_compact3(key >> 1), cz = (int)p2p_compact3(key >> 2);
        int32_t id = -1;
        if (lane < 27) {
            int x = cx + lane % 3 - 1, y = cy + (lane / 3) % 3 - 1, z = cz + lane / 9 - 1;
            if (x >= 0 && y >= 0 && z >= 0 && x < ng && y < ng && z < ng)
                id = find_key(src_keys, nbs, (int64_t)p2p_morton(x, y, z));
            found[b * 27 + lane] = id;
        }
        const unsigned any = __ballot_sync(P2P_FULL_MASK, id >= 0);
        int s = id >= 0 ? src_box_ptr[id + 1] - src_box_ptr[id] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(P2P_FULL_MASK, s, o);
        if (lane == 0) {
            cnt[b] = __popc(any);
            if (s) atomicAdd(&block_sum, (unsigned long long)s);
            if (b > 0 && box_keys[b - 1] >= box_keys[b]) *bad = 1;  // keys must strictly ascend
            if (!TWO && !((any >> 13) & 1u)) *bad = 1;               // a box must find itself
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && block_sum) atomicAdd(sum, block_sum);
}

// The found neighbours of every box in ascending order.
template <bool TWO>
__global__ void __launch_bounds__(kThreads)
    k_nbr_fill(const int32_t* __restrict__ found, int32_t nb, const int32_t* __restrict__ nbr_ptr,
               int32_t* __restrict__ nbr_idx, int32_t* __restrict__ nbr_self) {
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= nb) return;
    const int32_t id = lane < 27 ? found[b * 27 + lane] : -1;
    const int n = __popc(__ballot_sync(P2P_FULL_MASK, id >= 0));
    const int32_t v = warp_sort_asc(id >= 0 ? id : INT32_MAX, lane);
    if (lane < n) nbr_idx[nbr_ptr[b] + lane] = v;
    if (TWO) {
        // position of the source box of the target box's own cell (probe 13) in the sorted list
        const int32_t self = __shfl_sync(P2P_FULL_MASK, id, 13);
        const unsigned at = __ballot_sync(P2P_FULL_MASK, self >= 0 && v == self);
        if (lane == 0) nbr_self[b] = at ? __ffs(at) - 1 : -1;
    }
}

__global__ void k_keys_ascending(const int64_t* __restrict__ keys, int32_t n, int32_t* __restrict__ bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > 0 && i < n && keys[i - 1] >= keys[i]) *bad = 1;
}

// -------------------------------------------------------------------- plans --

__global__ void k_gather_xyz(const float* __restrict__ pts, const int32_t* __restrict__ perm, int64_t n,
                             float4* __restrict__ xs) {
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    int64_t j = perm[s];
    xs[s] = make_float4(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], 0.f);
}

// What plan creation has to know of the lists before it builds them (device, then host).
struct ListInfo {
    int32_t max_len, max_box;  // longest source list, largest box
    int32_t tails;             // lists just over one default chunk: a full item plus a short tail item
    int32_t packed;            // entries of all lists, each padded to 4
    int32_t items[3];          // work items with the chunk of each candidate tuning
    unsigned int status;       // nonzero: invalid CSR
    unsigned long long pairs;  // targets x sources of all boxes, and of the heaviest box
    unsigned long long heavy;
};

// Per target box: S_b, the length of its source list, and the size of the source box of its own cell (the sources
// that can sit at r = 0 from one of its targets).  Validates the CSR (ascending ids in range; a one-set structure
// lists each box itself, a two-set structure's nbr_self must point into the list or be -1).
__global__ void __launch_bounds__(kThreads)
    k_box_info(const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ src_box_ptr, int32_t nbs,
               const int32_t* __restrict__ nbr_ptr, const int32_t* __restrict__ nbr_idx,
               const int32_t* __restrict__ nbr_self, int32_t nb, int64_t nnz, int chunk0, int chunk1, int chunk2,
               int upper, int32_t* __restrict__ box_src, int32_t* __restrict__ list_len, int32_t* __restrict__ self_len,
               ListInfo* __restrict__ info) {
    const int32_t b = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    int64_t s = 0, s_up = 0;
    int32_t self_n = 0, own = 0;
    bool bad = false;
    if (b < nb) {
        const int32_t e0 = nbr_ptr[b], e1 = nbr_ptr[b + 1];
        int32_t self = -1;
        bool ok = e0 >= 0 && e1 >= e0 && e1 <= nnz && e1 - e0 <= 27;
        if (ok) {
            const int32_t want = nbr_self ? nbr_self[b] : -2;
            if (nbr_self && (want < -1 || want >= e1 - e0)) ok = false;
            int32_t prev = -1;
            for (int32_t e = e0; ok && e < e1; ++e) {
                const int32_t c = nbr_idx[e];
                if (c < 0 || c >= nbs || c <= prev) {
                    ok = false;
                    break;
                }
                prev = c;
                const int32_t sz = src_box_ptr[c + 1] - src_box_ptr[c];
                if (nbr_self ? (e - e0 == want) : (c == b)) {
                    self = e - e0;
                    self_n = sz;
                }
                s += sz;
                if (c >= b) s_up += sz;
            }
        }
        own = box_ptr[b + 1] - box_ptr[b];
        bad = !ok || (!nbr_self && self < 0) || own <= 0 || s > INT32_MAX - 4;
        if (bad) {
            s = 0;
            s_up = 0;
            self_n = 0;
        }
        box_src[b] = (int32_t)s;
        self_len[b] = self_n;
        list_len[b] = (int32_t)(upper ? s_up : s);
    }
    // one set of atomics per warp
    const int32_t len = (int32_t)(upper ? s_up : s);
    const bool tail = len > chunk0 && 3ll * len <= 4ll * chunk0;
    const int32_t max_len = __reduce_max_sync(P2P_FULL_MASK, len), max_own = __reduce_max_sync(P2P_FULL_MASK, own);
    const int32_t padded = __reduce_add_sync(P2P_FULL_MASK, (len + 3) & ~3);
    const int32_t i0 = __reduce_add_sync(P2P_FULL_MASK, (int32_t)(((int64_t)len + chunk0 - 1) / chunk0));
    const int32_t i1 = __reduce_add_sync(P2P_FULL_MASK, (int32_t)(((int64_t)len + chunk1 - 1) / chunk1));
    const int32_t i2 = __reduce_add_sync(P2P_FULL_MASK, (int32_t)(((int64_t)len + chunk2 - 1) / chunk2));
    const int tails = __popc(__ballot_sync(P2P_FULL_MASK, tail));
    const bool any_bad = __any_sync(P2P_FULL_MASK, bad);
    unsigned long long pairs = bad ? 0ull : (unsigned long long)own * (unsigned long long)s, heavy = pairs;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(P2P_FULL_MASK, pairs, o);
        heavy = max(heavy, __shfl_xor_sync(P2P_FULL_MASK, heavy, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&info->pairs, pairs);
        atomicMax(&info->heavy, heavy);
        atomicMax(&info->max_len, max_len);
        atomicMax(&info->max_box, max_own);
        if (tails) atomicAdd(&info->tails, tails);
        atomicAdd(&info->packed, padded);
        atomicAdd(&info->items[0], i0);
        atomicAdd(&info->items[1], i1);
        atomicAdd(&info->items[2], i2);
        if (any_bad) atomicOr(&info->status, P2P_DEV_BAD_INPUT);
    }
}

// Items and padded length of every box's list for the chosen chunk.
__global__ void k_list_sizes(const int32_t* __restrict__ list_len, int32_t nb, int chunk, int32_t* __restrict__ n_chunks,
                             int32_t* __restrict__ padded) {
    const int32_t b = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (b >= nb) return;
    const int32_t len = list_len[b];
    n_chunks[b] = (int32_t)(((int64_t)len + chunk - 1) / chunk);
    padded[b] = (len + 3) & ~3;
}

// Work-item records (unsorted) and their sort keys: larger cost (targets x
// sources) first.
__global__ void k_item_records(const int32_t* __restrict__ n_chunks, const int32_t* __restrict__ item_off,
                               const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ list_len,
                               const int32_t* __restrict__ self_len, const int32_t* __restrict__ pk_off, int32_t nb,
                               int chunk, int tg, int two_sets, bool fine, ItemRec* __restrict__ recs,
                               uint32_t* __restrict__ keys, int32_t* __restrict__ vals) {
    int32_t b = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (b >= nb) return;
    const int32_t c = n_chunks[b], o = item_off[b];
    const int32_t tb = box_ptr[b], nt = box_ptr[b + 1] - tb, S = list_len[b];
    const int32_t last = nt - ((nt - 1) / tg) * tg;  // targets of the last target group
    // the list in c near-equal items (multiples of 4 entries but the last, at most chunk each) rather than c - 1
    // full items and a short tail
    int32_t L = c > 1 ? (((S + c - 1) / c + 3) & ~3) : chunk;
    if ((c - 1) * L >= S) L = chunk;
    for (int32_t i = 0; i < c; ++i) {
        const int32_t s0 = i * L;
        ItemRec r;
        r.src_off = pk_off[b] + s0;
        r.ns = min(L, S - s0);
        r.tb = tb;
        r.nt = nt;
        // the own cell's sources lead the list; in a one-set plan they are the box's targets themselves
        r.m_end = max(0, min(r.ns, self_len[b] - s0)) | ((s0 == 0 && !two_sets) ? (1 << 16) : 0);
        r.map_full = p2p_lane_map(min(nt, tg), r.ns);
        r.map_last = p2p_lane_map(last, r.ns);
        r.b = b;
        recs[o + i] = r;
        keys[o + i] = fine ? cost_key<kFineCostBits>((int64_t)nt * r.ns) : cost_key<kCostBits>((int64_t)nt * r.ns);
        vals[o + i] = o + i;
    }
}

__global__ void k_item_gather(const ItemRec* __restrict__ recs, const int32_t* __restrict__ order, int64_t n,
                              ItemRec* __restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = recs[order[i]];
}

// Direct-kernel items: one per target box, its whole source list, lane maps for
// `lanes` lanes (passes of up to 4 * lanes targets), sort keys by decreasing cost.
__global__ void k_direct_items(const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ list_len,
                               const int32_t* __restrict__ self_len, const int32_t* __restrict__ pk_off, int32_t nb,
                               int lanes, ItemRec* __restrict__ recs, uint32_t* __restrict__ keys,
                               int32_t* __restrict__ vals) {
    const int32_t b = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (b >= nb) return;
    const int32_t tb = box_ptr[b], nt = box_ptr[b + 1] - tb, S = list_len[b];
    const int pass = 4 * lanes;
    const int32_t last = nt - ((nt - 1) / pass) * pass;
    ItemRec r;
    r.src_off = pk_off[b];
    r.ns = S;
    r.tb = tb;
    r.nt = nt;
    r.m_end = min(S, self_len[b]);
    r.map_full = p2p_lane_map(min(nt, pass), S, lanes, 8);
    r.map_last = p2p_lane_map(last, S, lanes, 8);
    r.b = b;
    recs[b] = r;
    keys[b] = cost_key<kFineCostBits>((int64_t)nt * S);
    vals[b] = b;
}

// One warp per target box: writes the box's source list -- the sources of its
// own cell first (the box itself in a one-set plan, the source box of the same
// cell in a two-set plan), then the other neighbour boxes in ascending id (the
// order the pair kernel's r = 0 mask relies on) -- as box-sorted source indices
// (nb_src, the index arrays of the indexing method, Sec. 3.2) and, for the
// redundant layout, as a copy of the coordinates (the repetition of Sec. 3.3).  xs
// and box_ptr are the SOURCE side.
__global__ void k_pack(const float4* __restrict__ xs, const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ nbr_ptr,
                       const int32_t* __restrict__ nbr_idx, const int32_t* __restrict__ nbr_self,
                       const int32_t* __restrict__ pk_off, int32_t nb, int upper, int32_t* __restrict__ nb_src,
                       float4* __restrict__ pk_xyz) {
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= nb) return;
    const int32_t e0 = nbr_ptr[b];
    int32_t ne = nbr_ptr[b + 1] - e0;
    const int32_t c = lane < ne ? nbr_idx[e0 + lane] : -1;
    int sp;
    if (nbr_self) {
        sp = nbr_self[b];  // -1: no source box in the own cell, the list keeps ascending order
    } else {
        const unsigned selfm = __ballot_sync(P2P_FULL_MASK, c == (int32_t)b);
        sp = selfm ? __ffs(selfm) - 1 : 0;
    }
    // full list: slot 0 <- own cell, slots 1..sp <- entries 0..sp-1, later slots unchanged;
    // upper list (own box and higher ids only): slot i <- entry sp + i
    int from = sp < 0 ? lane : (lane == 0 ? sp : (lane <= sp ? lane - 1 : lane));
    if (upper) {
        from = min(sp + lane, 31);
        ne -= sp;
    }
    const int32_t cs = __shfl_sync(P2P_FULL_MASK, c, from);
    int32_t start = 0, len = 0;
    if (lane < ne) {
        start = box_ptr[cs];
        len = box_ptr[cs + 1] - start;
    }
    int32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(P2P_FULL_MASK, incl, o);
        if (lane >= o) incl += y;
    }
    const int32_t excl = incl - len;
    const int32_t total = __shfl_sync(P2P_FULL_MASK, incl, 31);
    const int64_t base = pk_off[b];
    const int32_t padded = pk_off[b + 1] - pk_off[b];
    // neighbour after neighbour, each a run of consecutive indices (looking up the neighbour of every entry instead
    // took 55 us for the 15 M entries of the 2^20-point sphere at 32 points per box)
    for (int e = 0; e < ne; ++e) {
        const int32_t s0 = __shfl_sync(P2P_FULL_MASK, start, e), m = __shfl_sync(P2P_FULL_MASK, len, e);
        const int64_t to = base + __shfl_sync(P2P_FULL_MASK, excl, e);
        for (int32_t p = lane; p < m; p += 32) {
            const int32_t j = s0 + p;
            nb_src[to + p] = j;
            if (pk_xyz) pk_xyz[to + p] = xs[j];
        }
    }
    if (lane < padded - total) {
        nb_src[base + total + lane] = -1;
        if (pk_xyz) pk_xyz[base + total + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Pairs of target box b: n_b * S_b minus the (target, source) pairs of its own
// cell with identical coordinates (xt / box_ptr: targets; xs / src_box_ptr:
// sources; self_len / nbr_self locate the own cell's source box).
__global__ void k_pair_count(const float4* __restrict__ xt, const int32_t* __restrict__ box_ptr,
                             const float4* __restrict__ xs, const int32_t* __restrict__ src_box_ptr,
                             const int32_t* __restrict__ nbr_ptr, const int32_t* __restrict__ nbr_idx,
                             const int32_t* __restrict__ nbr_self, const int32_t* __restrict__ box_src, int32_t nb,
                             unsigned long long* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= nb) return;
    const int32_t t0 = box_ptr[b], t1 = box_ptr[b + 1];
    int32_t c = (int32_t)b;
    if (nbr_self) c = nbr_self[b] >= 0 ? nbr_idx[nbr_ptr[b] + nbr_self[b]] : -1;
    long long dup = 0;
    if (c >= 0) {
        const int32_t s0 = src_box_ptr[c], s1 = src_box_ptr[c + 1];
        for (int32_t i = t0 + lane; i < t1; i += 32) {
            float4 a = xt[i];
            for (int32_t j = s0; j < s1; ++j) {
                float4 q = xs[j];
                dup += (a.x == q.x && a.y == q.y && a.z == q.z) ? 1 : 0;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dup += __shfl_xor_sync(P2P_FULL_MASK, dup, o);
    if (lane == 0) {
        long long p = (long long)(t1 - t0) * (long long)box_src[b] - dup;
        atomicAdd(out, (unsigned long long)p);
    }
}

// Points (sorted position s) whose new coordinates fall in another grid cell
// than the coordinates the plan holds (same cell rule as the binning), and
// non-finite new coordinates.
__global__ void k_moved(const float* __restrict__ pts, const int32_t* __restrict__ perm,
                        const float4* __restrict__ xs, int64_t n, double lo0, double lo1, double lo2, double h, int ng,
                        unsigned long long* __restrict__ moved, int32_t* __restrict__ bad) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int64_t j = perm[s];
    const float x = pts[3 * j], y = pts[3 * j + 1], z = pts[3 * j + 2];
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) {
        *bad = 1;
        return;
    }
    const float4 o = xs[s];
    if (cell_of(x, lo0, h, ng) != cell_of(o.x, lo0, h, ng) || cell_of(y, lo1, h, ng) != cell_of(o.y, lo1, h, ng) ||
        cell_of(z, lo2, h, ng) != cell_of(o.z, lo2, h, ng))
        atomicAdd(moved, 1ull);
}

// Redundant layout: the per-box copies of the listed source coordinates from the box-sorted ones.
__global__ void k_repack_xyz(const float4* __restrict__ xs, const int32_t* __restrict__ nb_src, int64_t packed,
                             float4* __restrict__ pk_xyz) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= packed) return;
    const int32_t j = nb_src[p];
    pk_xyz[p] = j >= 0 ? xs[j] : make_float4(0.f, 0.f, 0.f, 0.f);
}

// Repetition layout: entries of the records of box b's targets, n_b (1 + S_b).
__global__ void k_rep_count(const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ box_src, int32_t nb,
                            int32_t* __restrict__ cnt) {
    const int32_t b = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (b < nb) cnt[b] = (box_ptr[b + 1] - box_ptr[b]) * (1 + box_src[b]);
}

// One warp per box: the records of its targets -- entry 0 the target's coordinates, entries 1 .. S_b a copy of
// the box's source list (own box first, then the other neighbour boxes in ascending id) with the sources'
// original indices, for the per-apply strength repack (the collection of Sec. 3.3, eq. 6, on the device).
__global__ void k_rep_fill(const float4* __restrict__ xs, const int32_t* __restrict__ perm,
                           const int32_t* __restrict__ box_ptr, const int32_t* __restrict__ box_src,
                           const int32_t* __restrict__ pk_off, const int32_t* __restrict__ nb_src,
                           const int32_t* __restrict__ rec_boff, int32_t nb, int64_t n, int32_t* __restrict__ rec_off,
                           float4* __restrict__ rec_xyz, int32_t* __restrict__ rec_src) {
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= nb) return;
    const int32_t tb = box_ptr[b], nt = box_ptr[b + 1] - tb, S = box_src[b], len = 1 + S;
    const int32_t* list = nb_src + pk_off[b];
    for (int32_t u = 0; u < nt; ++u) {
        const int64_t base = (int64_t)rec_boff[b] + (int64_t)u * len;
        if (lane == 0) {
            rec_off[tb + u] = (int32_t)base;
            rec_xyz[base] = xs[tb + u];
            rec_src[base] = -1;
        }
        for (int32_t p = lane; p < S; p += 32) {
            const int32_t j = list[p];
            rec_xyz[base + 1 + p] = xs[j];
            rec_src[base + 1 + p] = perm[j];
        }
    }
    if (b == nb - 1 && lane == 0) rec_off[n] = rec_boff[nb];
}

int ceil_log2(int v) {
    int b = 0;
    while ((1 << b) < v) ++b;
    return b;
}

inline int64_t head_blocks(int64_t n) { return (n + kThreads * kHeads - 1) / (kThreads * kHeads); }

struct BinLayout {
    uint64_t *keys, *keys_alt;
    int32_t *vals, *vals_alt, *heads, *first, *small;
    void *radix_ws, *scan_ws;
    size_t radix_bytes, bytes;
};

BinLayout bin_layout(int64_t n, void* work) {
    Carver c{static_cast<char*>(work), 0, (size_t)-1};
    BinLayout L;
    size_t m = (size_t)(n > 0 ? n : 1);
    L.keys = c.take<uint64_t>(m);
    L.keys_alt = c.take<uint64_t>(m);
    L.vals = c.take<int32_t>(m);
    L.vals_alt = c.take<int32_t>(m);
    L.heads = c.take<int32_t>((size_t)head_blocks((int64_t)m));
    L.first = c.take<int32_t>((size_t)head_blocks((int64_t)m));
    L.small = c.take<int32_t>(4);
    L.radix_bytes = radix_workspace_bytes(n);
    L.radix_ws = c.take<char>(L.radix_bytes);
    L.scan_ws = c.take<char>(scan_workspace_bytes(head_blocks((int64_t)m)));
    L.bytes = align_up(c.off, 256);
    return L;
}

// Morton keys of width K (32 bits hold grids of up to 1024 boxes per axis), their stable sort and the boxes.
// L.small: [0] non-finite flag, [1] number of boxes.
template <typename K>
cudaError_t bin_sorted(const BinLayout& L, const float* pts, int64_t n, const double lo[3], double h, int32_t ng, int bits,
                       int32_t* perm, int32_t* point_box, int64_t* box_keys, int32_t* box_ptr, cudaStream_t s) {
    AxisGrid g[3];
    for (int i = 0; i < 3; ++i) {
        g[i].lo = lo[i];
        g[i].h = h;
        g[i].lo_f = (float)lo[i];
        g[i].inv_h = (float)(1.0 / h);
        // grids so small or large that FP32 would flush or overflow keep the double division
        const bool plain = h > 1e-30 && h < 1e30 && fabs(lo[i]) < 1e30;
        g[i].slack = plain ? (float)((fabs(lo[i]) / h + 1.0) * 1.2e-7) : INFINITY;
    }
    K* keys = reinterpret_cast<K*>(L.keys);
    K* keys_alt = reinterpret_cast<K*>(L.keys_alt);
    k_keys<K><<<blocks_for(n, kThreads), kThreads, 0, s>>>(pts, n, g[0], g[1], g[2], ng, keys, L.vals, L.small);
    cudaError_t e = cudaGetLastError();
    bool in_alt = false;
    if (e == cudaSuccess) e = radix_sort_pairs(keys, L.vals, keys_alt, L.vals_alt, n, bits, L.radix_ws, L.radix_bytes, s, &in_alt);
    if (e != cudaSuccess) return e;
    const K* ks = in_alt ? keys_alt : keys;
    const int32_t* vs = in_alt ? L.vals_alt : L.vals;
    const int64_t blocks = head_blocks(n);
    k_heads<K><<<(unsigned)blocks, kThreads, 0, s>>>(ks, n, L.heads);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_exclusive_i32(L.heads, L.first, blocks, L.small + 1, L.scan_ws, s);
    if (e != cudaSuccess) return e;
    k_rle<K><<<(unsigned)blocks, kThreads, 0, s>>>(ks, vs, L.first, n, perm, point_box, box_keys, box_ptr);
    return cudaGetLastError();
}

struct NbrLayout {
    int32_t *cnt, *found, *bad;
    unsigned long long* sum;
    void* scan_ws;
    size_t bytes;
};

NbrLayout nbr_layout(int32_t nb, void* work) {
    Carver c{static_cast<char*>(work), 0, (size_t)-1};
    NbrLayout L;
    const size_t m = (size_t)(nb > 0 ? nb : 1);
    L.cnt = c.take<int32_t>(m);
    L.found = c.take<int32_t>(27 * m);
    L.sum = c.take<unsigned long long>(4);
    L.bad = reinterpret_cast<int32_t*>(L.sum + 1);
    L.scan_ws = c.take<char>(scan_workspace_bytes(nb));
    L.bytes = align_up(c.off, 256);
    return L;
}

bool tuning_valid(const p2p_tuning& t) {
    return t.chunk >= 32 && t.chunk <= 1024 && t.chunk % 32 == 0 && t.warps_per_cta >= 1 && t.warps_per_cta <= 16 &&
           t.target_group >= 32 && t.target_group <= 128 && t.target_group % 32 == 0 &&
           (t.warp_boxes == -2 || t.warp_boxes == -1 || t.warp_boxes == 0 || t.warp_boxes == 1 ||
            t.warp_boxes == 2 || t.warp_boxes == 4 || t.warp_boxes == 8 || t.warp_boxes == 16 || t.warp_boxes == 32);
}

// Default launch tuning; a plan whose caller leaves chunk and warps at zero may switch to kWideTuning or
// kNarrowTuning (see p2p_plan_create).
constexpr p2p_tuning kDefaultTuning{192, 8, 32, 0};
constexpr p2p_tuning kWideTuning{256, 6, 32, 0};
constexpr p2p_tuning kNarrowTuning{128, 8, 32, 0};

bool tuning_is_auto(const p2p_tuning* t) { return !t || (t->chunk == 0 && t->warps_per_cta == 0); }

p2p_tuning resolve_tuning(const p2p_tuning* t) {
    p2p_tuning r = kDefaultTuning;
    if (t) {
        if (t->chunk) r.chunk = t->chunk;
        if (t->warps_per_cta) r.warps_per_cta = t->warps_per_cta;
        if (t->target_group) r.target_group = t->target_group;
        r.warp_boxes = t->warp_boxes;
    }
    return r;
}

// Largest union the box-group kernel stages (sources; 24 bytes each in shared memory; its positions are 16-bit).
constexpr int32_t kGroupCapMax = 8192;

// The one-right-hand-side kernel of a plan left to choose (warp_boxes = 0), from the mean number of targets per box D,
// the number of boxes and the sources of all lists: > 0 boxes per warp of the direct kernel, -2 the box-group kernel (indexed layout only,
// other layouts take the staged pipeline), -1 the staged pipeline.
//
// The direct kernel with several boxes per warp does the least work per pair on sparse boxes, but a box there is a
// long serial chain on a few lanes: its heaviest boxes alone take 20 - 50 us at D = 3 - 9, so it pays once the rest
// of the chip needs that long too.  Few boxes are best cut into the staged pipeline's items, which spread one box over
// several warps.  Measured on GB300 (applies in us, Helmholtz on a sphere / in a cube, staged | group | direct with 1
// / 4 / 8 boxes per warp):
//   D = 1.6 (plate): 635 boxes 6.1 | 7.3 | 4.9 / 8.5 / 9.5; 10 319: 15 | 13 | 11 / 10 / 11.5, sixteen 11.7;
//             165 629: 148 | 124 | 93 / 34 / 26.5, sixteen 25.6
//   D = 2.3 (plate): 28 275: 31 | 26 | 21 / 16 / 16.5, sixteen 20; 453 351: 421 | 379 | 289 / 125 / 91, sixteen 102
//   D = 3.5:   1 140: 6.4 | 8.3 | 6.6 / 13.6 / 22.4       4 605: 9.3 | 9.4 | 8.8 / 14.3 / 23.2
//             18 924: 24 | 23 | 18.7 / 17.0 / 25          75 224: 82 | 71 | 56 / 37 / 43
//            285 361: 307 | 284 | 237 / 129 / 119
//   D = 6.2:   2 636: 10.3 | 10.7 | 10.7 / 32 / 51        10 263: 20 | 18.6 | 19.7 / 39 / 61
//             42 015: 60 | 54 | 53 / 58 / 79              165 248: 231 | 209 | 218 / 160 / 176
//   D = 8-9:   1 792: 11.7 | 11.5 | 15 / 50 / 92           7 197: 20 | 16.5 | 23 / 54 / 96
//             28 916: 58 | 51 | 56 / 77 / 110             62 577: 107 | 97 | 102 / 102 / 133 (Laplace 91 | 81 | 81 / 70)
//            131 431: 218 | 197 | 219 / 188 / 225
//   D = 10.8: 97 091: 224 | 201 | 241 / 262 / 309
//   D = 14:    1 201: 12.9 | 16 | 25 / 77 / 152             4 829: 25 | 21 | 39    18 863: 72 | 66 | 78
//   D = 20:      784: 13.8 | 25 | 48                        3 296: 31 | 35 | 54    13 599: 88 | 85 | 102
//   cube, D = 9: 6 859: 30 | 25 | 31 / 86 / 156; D = 16: 1 000: 17 | 27, 17 576: 118 | 98; D = 21: 3 375: 40 | 45,
//   12 167: 147 | 151; D = 32 (4 096 boxes): 122 | 137
// Laplace gives the same ranking at about two thirds of the times, with several boxes per warp earlier (plan_warp_boxes).
//
// Which of two kernels is ahead also depends on the mean list length L (L = 12 - 15 D on a surface, up to 27 D in a
// volume).  Applies in a loop, staging and launches included:
//   eight | four boxes per warp   L = 27: 79 346 boxes 35.9 | 35.9 (Laplace 29.7 | 31.6), 126 626 46 | 48 (37.7 | 41.8); L = 30:
//             92 350 41 | 37, 148 652 48 | 50 (39.9 | 44.1); L = 40: 117 269 58 | 55; L = 45: 138 941 73 | 79, 198 460 108 | 111;
//             L = 53: 162 659 98 | 97; L = 77: 225 809 134 | 127; L = 105: 245 458 211 | 202
//   sixteen | eight               L = 15, D = 2.0: 199 650 42 | 40, 349 478 60 | 62 (Laplace, redundant layout 83 | 88)
//   group | staged                D = 18, surface: 1 108 24.6 | 18.5, 2 229 24.3 | 19.3, 4 579 31.6 | 32.2; cube: 1 000 29.9 | 15.9,
//             1 331 30.2 | 18.5, 2 197 27.6 | 28.9, 4 913 47 | 45, 6 859 57 | 62
//             D = 20 - 23, sphere: 2 259 32 | 27, 4 626 46 | 48 (Laplace 31.4 | 35.8), 6 970 77 | 58, 10 718 92 | 83 (two blocks
//             per SM: 304 groups are a wave), 19 332 137 | 144 (89 | 98); plate: 18 225 87 | 96 (56 | 64), 45 369 200 | 231;
//             cube: 4 913 69 | 63, 6 859 109 | 91, 10 648 132 | 135, 29 791 387 | 415
// On surfaces of 1 000 - 4 000 boxes at D = 12 - 19.5 the staged pipeline would be up to 1.3 times as fast; the box-group
// kernel is kept there, which callers of such plans see in p2p_plan_info and batches of them build on.
int32_t auto_warp_boxes(int64_t n, int32_t nb, int64_t sources) {
    if (nb <= 0) return -1;
    const double d = (double)n / nb, len = (double)sources / nb;
    const bool volume = len > 300.0;
    if (d > 24.0) return -1;
    if (d > 20.0) return nb >= (volume ? 10000 : 4000) ? -2 : -1;
    if (d > 12.0) return nb >= 4000 || (nb >= (volume ? 2000 : 1000) && d <= 19.5) ? -2 : -1;
    if (nb < 2500) return d <= 2.5 ? 1 : -1;
    if (d <= 1.3) return nb < 15000 ? 4 : 32;
    if (d <= 1.9 || (d <= 2.05 && len <= 16.0 && nb >= 250000)) return nb < 15000 ? 4 : 16;
    if (d <= 2.5) return nb < 15000 ? 4 : 8;
    if (d <= 5.2) return nb < 15000 ? 1 : (len <= 50.0 && nb >= (len <= 28.0 ? 75000 : 120000) ? 8 : 4);
    if (d <= 7.0) return nb < 45000 ? 1 : 4;
    return d <= 9.1 && nb >= 55000 ? 4 : -2;
}

// The same for a plan's kernel function and layout.  A Laplace pair costs two thirds of a Helmholtz one, so a box's chain
// on a few lanes hides earlier.  Measured (us):
//   four | one box per warp   D = 6.2: 40 303 boxes 34 | 40, 39 595 (L = 82) 44 | 46, 20 978 27.6 | 25.6
//   eight | four              D = 3.6, L = 43: 111 854 43 | 46
//   four | group              D = 8, L = 71: 31 317 37 | 42, 50 163 48 | 60; L = 106: 31 311 49 | 46, 50 124 62 | 71; L = 202: 29 788
//                             77 | 66, 50 633 97 | 103; D = 9, L = 80: 44 516 53 | 57; L = 120: 110 529 146 | 160; D = 10, L = 89:
//                             24 964 44 | 38, 39 998 54 | 54, 70 224 78 | 91; L = 133: 71 093 122 | 114
//   four | staged (redundant) D = 8, L = 71: 31 317 40 | 48; L = 106: 50 124 93 | 83; D = 10, L = 90: 39 998 72 | 67, 99 852 148 | 158
int32_t plan_warp_boxes(int64_t n, int32_t nb, int64_t sources, p2p_kernel kernel, p2p_layout layout) {
    const int32_t wb = auto_warp_boxes(n, nb, sources);
    const double d = (double)n / (nb > 0 ? nb : 1), len = (double)sources / (nb > 0 ? nb : 1);
    if (kernel == P2P_LAPLACE) {
        if (wb == 1 && d > 5.2 && nb >= 24000) return 4;
        if (wb == 4 && d > 2.5 && d <= 5.2 && len <= 45.0 && nb >= 100000) return 8;
        if (wb == -2 && d <= 12.0) {
            const bool indexed = layout == P2P_LAYOUT_INDEXED;
            if (len <= 95.0 && (d <= 8.5 ? nb >= 30000 : d <= 10.5 && nb >= (indexed ? 40000 : 55000))) return 4;
            if (indexed && (d <= 8.5 ? nb >= 45000 : d <= 9.2 && len <= 125.0 && nb >= 55000)) return 4;
        }
    }
    return wb == -2 && layout != P2P_LAYOUT_INDEXED ? -1 : wb;
}

// Whether the kernel that plan_warp_boxes names would wait for the heaviest box.  There a box stays on one warp, or on
// 32 / wb lanes of one, while the staged pipeline cuts it into items, so a cluster in an otherwise even geometry decides
// the apply, whatever the mean occupancy.  The direct kernel takes ~3.7 ns per pair of a box's share of the warp, the
// staged one 1.1 - 1.7 ns per box of the plan; the box-group kernel is behind once its heaviest box is worth 2.5 times the
// average warp and long by itself (24 576 pairs take it ~40 us).  Measured (us), spheres with patches of 3, 6 and 12
// times the mean density:
//   direct / staged   25 773 boxes of 3.9 74 / 37, 158 / 38, 413 / 48; 103 990 of 3.8 93 / 115, 194 / 116, 491 / 127;
//                     259 512 of 3.9 208 / 280, 397 / 281, 1201 / 286; 125 720 of 8.0 386 / 212, 858 / 218, 2453 / 246
//   group / staged    47 636 boxes of 8.4 101 / 92, 165 / 99, 372 / 132; 10 965 of 9.1 60 / 38, 118 / 51, 352 / 80
// and clustered assemblies, group / staged: 3 771 boxes of 8 193 / 32, 34 136 of 11.7 434 / 143, 84 640 of 11.8 800 / 335;
// direct / staged: 123 825 of 8.1 2317 / 332, in the redundant layout with the Laplace kernel 1699 / 234.
bool heaviest_decides(int32_t wb, const ListInfo& info, int32_t nb, int sms) {
    const double heavy = (double)info.heavy;
    if (wb > 0) return heavy * wb > 61.0 / sms * nb + 4096.0;
    return heavy > 24576.0 && heavy * (24.0 * sms) > 2.5 * (double)info.pairs;
}

struct PlanLayout {
    p2p_plan p;  // pointers only
    int32_t *n_chunks, *item_off, *padded, *maxes, *list_len, *self_len;
    ListInfo* info;
    void* scan_ws;
    // item-sort scratch (aliases the strength staging buffer when it is large enough)
    ItemRec* recs;
    uint32_t *keys, *keys_alt;
    int32_t *vals, *vals_alt;
    void* radix_ws;
    size_t radix_bytes, bytes;
};

// Sizes of a plan: n targets in nb boxes, n_src sources in nbs boxes (two_sets), sources = sum of S_b.
PlanLayout plan_layout(int64_t n, int32_t nb, int64_t n_src, int32_t nbs, bool two_sets, int64_t sources, int64_t nnz,
                       p2p_layout layout, int32_t max_nrhs, const p2p_tuning& t, void* ws, int64_t records = 0) {
    Carver c{static_cast<char*>(ws), 0, (size_t)-1};
    PlanLayout L;
    memset(&L.p, 0, sizeof(L.p));
    size_t m = (size_t)(n > 0 ? n : 1), mb = (size_t)(nb > 0 ? nb : 1);
    size_t ms = (size_t)(n_src > 0 ? n_src : 1), mbs = (size_t)(nbs > 0 ? nbs : 1);
    // room for the items of the narrowest chunk a plan may switch to
    const int sizing_chunk = t.chunk < kNarrowTuning.chunk ? t.chunk : kNarrowTuning.chunk;
    const size_t max_items = (size_t)(sources / sizing_chunk) + mb + 1;
    const size_t list_bound = (size_t)sources + 3 * mb + 4;
    const bool red = layout == P2P_LAYOUT_REDUNDANT;
    L.p.status = c.take<unsigned int>(4);
    L.p.scratch64 = c.take<long long>(4);
    L.p.xs = c.take<float4>(m);
    L.p.xs_src = two_sets ? c.take<float4>(ms) : L.p.xs;
    L.p.box_src = c.take<int32_t>(mb);
    L.p.items = c.take<ItemRec>(max_items);
    L.p.ditems = c.take<ItemRec>(mb);
    if (layout == P2P_LAYOUT_INDEXED && (t.warp_boxes == -2 || (t.warp_boxes == 0 && auto_warp_boxes(n, nb, sources) == -2))) {
        // box-group kernel tables (requested, or the plan's own choice)
        const size_t ngr = (mb + kGroupBoxes - 1) / kGroupBoxes;
        L.p.g_union = c.take<int32_t>(ngr * kGroupBoxes * 27);
        L.p.g_nunion = c.take<int32_t>(ngr);
        L.p.g_order = c.take<int32_t>(ngr);
        L.p.g_pos = c.take<int16_t>(list_bound);
        L.p.g_mend = c.take<int32_t>(mb);
        L.p.g_map = c.take<int32_t>(2 * mb);
        L.p.g_morder = c.take<int32_t>(ngr * kGroupBoxes);
        L.p.g_copy = c.take<int4>(ngr * kGroupBoxes * 27);
    }
    L.p.pk_off = c.take<int32_t>(mb + 1);
    L.p.nb_src = c.take<int32_t>(list_bound);
    L.p.pk_xyz = red ? c.take<float4>(list_bound) : nullptr;
    const bool rep = layout == P2P_LAYOUT_REPETITION;
    const size_t mr = (size_t)(records > 0 ? records : 1);
    L.p.rec_off = rep ? c.take<int32_t>(m + 1) : nullptr;
    L.p.rec_boff = rep ? c.take<int32_t>(mb + 1) : nullptr;
    L.p.rec_xyz = rep ? c.take<float4>(mr) : nullptr;
    L.p.rec_src = rep ? c.take<int32_t>(mr) : nullptr;
    size_t lam_rows = ms;
    if (rep && mr > lam_rows) lam_rows = mr;
    // rows of max_nrhs strengths (as they come, or packed), or sorted rows of the padded blocks of p2p_multi.cu
    size_t lam_count = lam_rows * (size_t)max_nrhs;
    if (lam_count < ms * (size_t)p2p_multi_columns(max_nrhs)) lam_count = ms * (size_t)p2p_multi_columns(max_nrhs);
    // ... or the coordinate gradient's rows (lambda, g)
    if (!two_sets && lam_count < 2 * m * (size_t)max_nrhs) lam_count = 2 * m * (size_t)max_nrhs;
    const size_t lam_bytes = lam_count * sizeof(float2);
    L.p.lam_buf = c.take<float2>(lam_count);
    const size_t tc_bytes = p2p_tc_pack_bytes((int64_t)ms, max_nrhs);
    if (tc_bytes) {
        const size_t blocks = (size_t)p2p_tc_block_count((int32_t)mb), entries = p2p_tc_entry_bound(sources, nnz);
        L.p.tc_off = c.take<int32_t>(blocks + 1);
        L.p.tc_ustart = c.take<int32_t>(blocks + 1);
        L.p.tc_ecount = c.take<int32_t>(blocks);
        L.p.tc_unit_block = c.take<int32_t>((size_t)p2p_tc_unit_bound((int64_t)m, (int32_t)mb));
        L.p.tc_gid = c.take<int32_t>(entries);
        L.p.tc_bits = c.take<uint32_t>(entries);
        L.p.tc_masks = c.take<uint32_t>(entries * 16);
        L.p.tc_member = c.take<uint8_t>(m);
        L.p.tc_counter = c.take<unsigned int>(2);
        const bool by_box = p2p_tcb_planned((int64_t)m, max_nrhs);
        const size_t box_bytes = by_box ? p2p_tcb_pack_bytes((int64_t)ms, (int32_t)mbs, max_nrhs) : 0;
        L.p.tc_pack = c.take<unsigned char>(tc_bytes > box_bytes ? tc_bytes : box_bytes);
        L.p.tcb_gstart = by_box ? c.take<int32_t>(mbs + 1) : nullptr;
        L.p.tcb_glist_off = by_box ? c.take<int32_t>(mb + 1) : nullptr;
        L.p.tcb_gcount = by_box ? c.take<int32_t>(mb) : nullptr;
        L.p.tcb_glist = by_box ? c.take<int32_t>(p2p_tcb_list_bound(sources, nnz, (int32_t)mb)) : nullptr;
    }
    const size_t mx = mb > mbs ? mb : mbs;
    L.n_chunks = c.take<int32_t>(mx);
    L.list_len = c.take<int32_t>(mb);
    L.self_len = c.take<int32_t>(mb);
    L.item_off = c.take<int32_t>(mb + 1);
    L.padded = c.take<int32_t>(mb);
    L.maxes = c.take<int32_t>(4);
    L.info = c.take<ListInfo>(1);
    L.scan_ws = c.take<char>(scan_workspace_bytes((int64_t)mx));
    // sort scratch: inside lam_buf if it fits, else after everything else
    Carver sc{reinterpret_cast<char*>(L.p.lam_buf), 0, lam_bytes};
    sc.take<ItemRec>(max_items);
    sc.take<uint32_t>(max_items);
    sc.take<uint32_t>(max_items);
    sc.take<int32_t>(max_items);
    sc.take<int32_t>(max_items);
    L.radix_bytes = radix_workspace_bytes((int64_t)max_items);
    sc.take<char>(L.radix_bytes);
    Carver& cs = (sc.off <= lam_bytes) ? sc : c;
    if (&cs == &sc) sc.off = 0;
    L.recs = cs.take<ItemRec>(max_items);
    L.keys = cs.take<uint32_t>(max_items);
    L.keys_alt = cs.take<uint32_t>(max_items);
    L.vals = cs.take<int32_t>(max_items);
    L.vals_alt = cs.take<int32_t>(max_items);
    L.radix_ws = cs.take<char>(L.radix_bytes);
    L.bytes = align_up(c.off, 256);
    return L;
}

// Everything a plan is made from: the target side (points, perm, boxes), the
// source side (the same arrays for a one-set plan) and the target-to-source
// neighbour CSR.
struct PlanInput {
    const float* pts;
    int64_t n;
    const int32_t* perm;
    const int32_t* box_ptr;
    int32_t nb;
    const float* src_pts;
    int64_t n_src;
    const int32_t* src_perm;
    const int32_t* src_box_ptr;
    int32_t nbs;
    const int32_t* nbr_ptr;
    const int32_t* nbr_idx;
    const int32_t* nbr_self;  // NULL for one-set plans
    int64_t nnz;
    int64_t sources;
    bool two_sets;
};

p2p_status check_sizes(int64_t n, int32_t nb, int64_t n_src, int32_t nbs, int64_t sources, p2p_layout layout,
                       int32_t max_nrhs, bool two_sets) {
    if (n < 0 || n >= INT32_MAX || nb < 0 || nb > n || n_src < 0 || n_src >= INT32_MAX || nbs < 0 || nbs > n_src ||
        sources < 0 || sources >= INT32_MAX || max_nrhs < 1 || max_nrhs > 256)
        return P2P_ERR_INVALID;
    if (layout != P2P_LAYOUT_INDEXED && layout != P2P_LAYOUT_REDUNDANT && layout != P2P_LAYOUT_SYMMETRIC &&
        layout != P2P_LAYOUT_REPETITION)
        return P2P_ERR_INVALID;
    if (two_sets && (layout == P2P_LAYOUT_SYMMETRIC || layout == P2P_LAYOUT_REPETITION)) return P2P_ERR_UNSUPPORTED;
    if (layout == P2P_LAYOUT_REPETITION && max_nrhs != 1) return P2P_ERR_UNSUPPORTED;
    return P2P_OK;
}

p2p_status plan_create(p2p_plan** plan, const PlanInput& in, p2p_kernel kernel, float k, p2p_layout layout,
                       int32_t max_nrhs, const p2p_tuning* tuning, void* workspace, size_t workspace_bytes,
                       cudaStream_t s);

}  // namespace

// ===================================================================== C ABI ==

extern "C" {

P2P_API int32_t p2p_version(void) { return 100; }

P2P_API const char* p2p_status_string(p2p_status s) {
    switch (s) {
        case P2P_OK: return "ok";
        case P2P_ERR_INVALID: return "invalid argument or input";
        case P2P_ERR_WORKSPACE: return "workspace too small";
        case P2P_ERR_CUDA: return "CUDA error";
        case P2P_ERR_TIMEOUT: return "device-side wait timed out";
        case P2P_ERR_UNSUPPORTED: return "unsupported";
        case P2P_ERR_ALLOC: return "host allocation failed";
        case P2P_ERR_STALE: return "a point left its leaf box: rebuild the plan";
    }
    return "unknown status";
}

P2P_API const char* p2p_last_error_string(void) { return g_last_error; }

P2P_API p2p_status p2p_bin_workspace_size(int64_t n, size_t* bytes) {
    if (!bytes || n < 0 || n >= INT32_MAX) return P2P_ERR_INVALID;
    *bytes = bin_layout(n, nullptr).bytes;
    return P2P_OK;
}

P2P_API p2p_status p2p_bin_points(const float* pts, int64_t n, const double lo[3], double h, int32_t ng,
                                  int32_t* perm, int32_t* point_box, int64_t* box_keys, int32_t* box_ptr,
                                  int32_t* num_boxes, void* work, size_t work_bytes, p2p_stream_t stream) {
    if (n < 0 || n >= INT32_MAX || !lo || !num_boxes || !box_ptr || !(h > 0.0) || !isfinite(h) || ng < 1 ||
        ng > (1 << 21))
        return P2P_ERR_INVALID;
    if (!isfinite(lo[0]) || !isfinite(lo[1]) || !isfinite(lo[2])) return P2P_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    *num_boxes = 0;
    if (n == 0) {
        P2P_TRY_CUDA(cudaMemsetAsync(box_ptr, 0, sizeof(int32_t), s), "p2p_bin_points");
        P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_bin_points");
        return P2P_OK;
    }
    if (!pts || !perm || !point_box || !box_keys || !work) return P2P_ERR_INVALID;
    if (((uintptr_t)pts & 3) || ((uintptr_t)work & 255)) return P2P_ERR_INVALID;
    BinLayout L = bin_layout(n, work);
    if (work_bytes < L.bytes) return P2P_ERR_WORKSPACE;

    P2P_TRY_CUDA(cudaMemsetAsync(L.small, 0, 4 * sizeof(int32_t), s), "p2p_bin_points");
    const int bits = 3 * ceil_log2(ng);
    const cudaError_t e = bits <= 32 ? bin_sorted<uint32_t>(L, pts, n, lo, h, ng, bits, perm, point_box, box_keys, box_ptr, s)
                                     : bin_sorted<uint64_t>(L, pts, n, lo, h, ng, bits, perm, point_box, box_keys, box_ptr, s);
    P2P_TRY_CUDA(e, "p2p_bin_points");
    int32_t host[2] = {0, 0};
    P2P_TRY_CUDA(cudaMemcpyAsync(host, L.small, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, s), "p2p_bin_points");
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_bin_points");
    if (host[0]) return P2P_ERR_INVALID;
    *num_boxes = host[1];  // total of the head flags = number of non-empty boxes
    return P2P_OK;
}

P2P_API p2p_status p2p_neighbors_workspace_size(int32_t num_boxes, size_t* bytes) {
    if (!bytes || num_boxes < 0) return P2P_ERR_INVALID;
    *bytes = nbr_layout(num_boxes, nullptr).bytes;
    return P2P_OK;
}

}  // extern "C"

namespace {

// Neighbour CSR of nb target boxes over nbs source boxes (the same boxes for a one-set structure).
p2p_status build_neighbors(const int64_t* box_keys, int32_t num_boxes, const int64_t* src_keys,
                           const int32_t* src_box_ptr, int32_t num_src, int32_t ng, int32_t* nbr_ptr,
                           int32_t* nbr_idx, int32_t* nbr_self, int64_t* nnz, int64_t* sources, void* work,
                           size_t work_bytes, cudaStream_t s, bool two) {
    if (num_boxes < 0 || num_src < 0 || ng < 1 || ng > (1 << 21) || !nbr_ptr || !nnz || !sources)
        return P2P_ERR_INVALID;
    *nnz = 0;
    *sources = 0;
    if (num_boxes == 0) {
        P2P_TRY_CUDA(cudaMemsetAsync(nbr_ptr, 0, sizeof(int32_t), s), "p2p_build_neighbors");
        P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_build_neighbors");
        return P2P_OK;
    }
    if (!box_keys || !src_keys || !src_box_ptr || !nbr_idx || !work || ((uintptr_t)work & 255)) return P2P_ERR_INVALID;
    if (two && !nbr_self) return P2P_ERR_INVALID;
    if ((int64_t)num_boxes * 27 >= INT32_MAX) return P2P_ERR_UNSUPPORTED;
    NbrLayout L = nbr_layout(num_boxes, work);
    if (work_bytes < L.bytes) return P2P_ERR_WORKSPACE;
    // [0] sources, [1] flag of invalid keys, [2] (filled below) list entries
    P2P_TRY_CUDA(cudaMemsetAsync(L.sum, 0, 4 * sizeof(unsigned long long), s), "p2p_build_neighbors");
    const unsigned wblocks = blocks_for((int64_t)num_boxes * 32, kThreads);
    if (two) {
        if (num_src > 1) {
            k_keys_ascending<<<blocks_for(num_src, kThreads), kThreads, 0, s>>>(src_keys, num_src, L.bad);
            P2P_CHECK_LAUNCH("p2p_build_neighbors_st/keys");
        }
        k_nbr_find<true><<<wblocks, kThreads, 0, s>>>(box_keys, num_boxes, src_keys, num_src, src_box_ptr, ng, L.cnt,
                                                      L.found, L.sum, L.bad);
    } else {
        k_nbr_find<false><<<wblocks, kThreads, 0, s>>>(box_keys, num_boxes, src_keys, num_src, src_box_ptr, ng, L.cnt,
                                                       L.found, L.sum, L.bad);
    }
    P2P_CHECK_LAUNCH("p2p_build_neighbors/find");
    P2P_TRY_CUDA(scan_exclusive_i32(L.cnt, nbr_ptr, num_boxes, nbr_ptr + num_boxes, L.scan_ws, s),
                 "p2p_build_neighbors/scan");
    if (two) k_nbr_fill<true><<<wblocks, kThreads, 0, s>>>(L.found, num_boxes, nbr_ptr, nbr_idx, nbr_self);
    else k_nbr_fill<false><<<wblocks, kThreads, 0, s>>>(L.found, num_boxes, nbr_ptr, nbr_idx, nullptr);
    P2P_CHECK_LAUNCH("p2p_build_neighbors/fill");
    P2P_TRY_CUDA(cudaMemcpyAsync(L.sum + 2, nbr_ptr + num_boxes, sizeof(int32_t), cudaMemcpyDeviceToDevice, s),
                 "p2p_build_neighbors");
    unsigned long long host[3] = {0, 0, 0};
    P2P_TRY_CUDA(cudaMemcpyAsync(host, L.sum, sizeof(host), cudaMemcpyDeviceToHost, s), "p2p_build_neighbors");
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_build_neighbors");
    const bool bad = (uint32_t)host[1] != 0;
    const int32_t total = (int32_t)host[2];
    const unsigned long long src = host[0];
    if (bad) return P2P_ERR_INVALID;
    *nnz = total;
    *sources = (int64_t)src;
    return P2P_OK;
}

// Entries of the repetition layout's records, sum over boxes of n_b (1 + S_b), from the box pointers and the
// neighbour lists copied to the host.
p2p_status repetition_records(const int32_t* box_ptr, int32_t nb, const int32_t* nbr_ptr, const int32_t* nbr_idx,
                              int64_t* records, cudaStream_t s) {
    *records = 0;
    if (nb <= 0) return P2P_OK;
    int32_t* hb = (int32_t*)malloc(sizeof(int32_t) * ((size_t)nb + 1) * 2);
    if (!hb) return P2P_ERR_ALLOC;
    int32_t* hp = hb + nb + 1;
    cudaError_t e = cudaMemcpyAsync(hb, box_ptr, sizeof(int32_t) * ((size_t)nb + 1), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hp, nbr_ptr, sizeof(int32_t) * ((size_t)nb + 1), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    int32_t* hi = nullptr;
    const int64_t nnz = e == cudaSuccess ? hp[nb] : 0;
    if (e == cudaSuccess && (nnz < 0 || nnz > 27ll * nb || hp[0] != 0)) {
        free(hb);
        return P2P_ERR_INVALID;
    }
    if (e == cudaSuccess && nnz > 0) {
        hi = (int32_t*)malloc(sizeof(int32_t) * (size_t)nnz);
        if (!hi) {
            free(hb);
            return P2P_ERR_ALLOC;
        }
        e = cudaMemcpyAsync(hi, nbr_idx, sizeof(int32_t) * (size_t)nnz, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) {
        free(hb);
        free(hi);
        set_cuda_error(e, "p2p_repetition_records");
        return P2P_ERR_CUDA;
    }
    int64_t total = 0;
    p2p_status st = P2P_OK;
    for (int32_t b = 0; b < nb && st == P2P_OK; ++b) {
        int64_t sb = 0;
        for (int32_t q = hp[b]; q < hp[b + 1]; ++q) {
            const int32_t c = hi[q];
            if (c < 0 || c >= nb) {
                st = P2P_ERR_INVALID;
                break;
            }
            sb += hb[c + 1] - hb[c];
        }
        total += (int64_t)(hb[b + 1] - hb[b]) * (1 + sb);
    }
    free(hb);
    free(hi);
    if (st != P2P_OK) return st;
    *records = total;
    return P2P_OK;
}

p2p_status plan_create(p2p_plan** plan, const PlanInput& in, p2p_kernel kernel, float k, p2p_layout layout,
                       int32_t max_nrhs, const p2p_tuning* tuning, void* workspace, size_t workspace_bytes,
                       cudaStream_t s) {
    if (!plan) return P2P_ERR_INVALID;
    *plan = nullptr;
    p2p_status st = check_sizes(in.n, in.nb, in.n_src, in.nbs, in.sources, layout, max_nrhs, in.two_sets);
    if (st != P2P_OK) return st;
    p2p_tuning t = resolve_tuning(tuning);
    if (!tuning_valid(t)) return P2P_ERR_INVALID;
    const int32_t nb = in.nb;
    const int64_t n = in.n;
    if (kernel != P2P_HELMHOLTZ && kernel != P2P_LAPLACE) return P2P_ERR_INVALID;
    if (!isfinite(k)) return P2P_ERR_INVALID;
    if ((n > 0 && nb < 1) || (n == 0 && nb != 0)) return P2P_ERR_INVALID;
    if ((in.n_src > 0 && in.nbs < 1) || (in.n_src == 0 && in.nbs != 0)) return P2P_ERR_INVALID;
    if (in.two_sets ? (in.nnz < 0 || in.nnz > 27ll * nb) : (in.nnz < nb || in.nnz > 27ll * nb))
        return P2P_ERR_INVALID;
    if (n > 0 && (!in.pts || !in.perm || !in.box_ptr || !in.nbr_ptr || (in.nnz > 0 && !in.nbr_idx)))
        return P2P_ERR_INVALID;
    if (in.two_sets && n > 0 && (!in.nbr_self || (in.n_src > 0 && (!in.src_pts || !in.src_perm || !in.src_box_ptr))))
        return P2P_ERR_INVALID;
    if (!workspace || ((uintptr_t)workspace & 255) || ((uintptr_t)in.pts & 3) || ((uintptr_t)in.src_pts & 3))
        return P2P_ERR_INVALID;
    int64_t records = 0;
    if (layout == P2P_LAYOUT_REPETITION) {
        const p2p_status rs = repetition_records(in.box_ptr, nb, in.nbr_ptr, in.nbr_idx, &records, s);
        if (rs != P2P_OK) return rs;
        if (records >= INT32_MAX) return P2P_ERR_UNSUPPORTED;
    }
    PlanLayout L = plan_layout(n, nb, in.n_src, in.nbs, in.two_sets, in.sources, in.nnz, layout, max_nrhs, t,
                               workspace, records);
    if (workspace_bytes < L.bytes) return P2P_ERR_WORKSPACE;
    p2p_plan* p = (p2p_plan*)malloc(sizeof(p2p_plan));
    if (!p) return P2P_ERR_ALLOC;
    *p = L.p;
    p->n = n;
    p->nb = nb;
    p->two_sets = in.two_sets ? 1 : 0;
    p->n_src = in.n_src;
    p->nbs = in.nbs;
    p->nnz = in.nnz;
    p->sources = in.sources;
    p->kernel = kernel;
    p->k = kernel == P2P_LAPLACE ? 0.f : k;
    p->layout = layout;
    p->max_nrhs = max_nrhs;
    p->tune = t;
    p->pts = in.pts;
    p->perm = in.perm;
    p->box_ptr = in.box_ptr;
    p->nbr_ptr = in.nbr_ptr;
    p->nbr_idx = in.nbr_idx;
    p->src_pts = in.src_pts;
    p->src_perm = in.src_perm;
    p->src_box_ptr = in.src_box_ptr;
    p->nbr_self = in.two_sets ? in.nbr_self : nullptr;
    p->n_items = 0;
    p->max_chunks = 0;
    p->max_box = 0;
    p->packed = 0;
    p->tc_wait_polls = -1;
    p->records = records;
#define FAIL_CUDA(expr, where)                 \
    do {                                       \
        cudaError_t e_ = (expr);               \
        if (e_ != cudaSuccess) {               \
            set_cuda_error(e_, where);         \
            free(p);                           \
            return P2P_ERR_CUDA;               \
        }                                      \
    } while (0)
    FAIL_CUDA(cudaMemsetAsync(p->status, 0, 4 * sizeof(unsigned int), s), "p2p_plan_create");
    if (n == 0) {
        FAIL_CUDA(cudaStreamSynchronize(s), "p2p_plan_create");
        *plan = p;
        return P2P_OK;
    }
    k_gather_xyz<<<blocks_for(n, kThreads), kThreads, 0, s>>>(in.pts, in.perm, n, p->xs);
    FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/gather");
    if (in.two_sets && in.n_src > 0) {
        k_gather_xyz<<<blocks_for(in.n_src, kThreads), kThreads, 0, s>>>(in.src_pts, in.src_perm, in.n_src, p->xs_src);
        FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/gather_sources");
    }
    // The lists' sizes for every tuning the plan may take, read back once; nothing is built from an invalid CSR.
    const int upper = layout == P2P_LAYOUT_SYMMETRIC;
    const bool choose = tuning_is_auto(tuning);
    const p2p_tuning* candidates[3] = {&t, choose ? &kWideTuning : &t, choose ? &kNarrowTuning : &t};
    FAIL_CUDA(cudaMemsetAsync(L.info, 0, sizeof(ListInfo), s), "p2p_plan_create");
    k_box_info<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(
        in.box_ptr, p->src_box_ptr, p->nbs, in.nbr_ptr, in.nbr_idx, p->nbr_self, nb, in.nnz, candidates[0]->chunk,
        candidates[1]->chunk, candidates[2]->chunk, upper, p->box_src, L.list_len, L.self_len, L.info);
    FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/box_info");
    ListInfo info;
    int sms = 0, dev = 0;
    FAIL_CUDA(cudaGetDevice(&dev), "p2p_plan_create");
    FAIL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "p2p_plan_create");
    FAIL_CUDA(cudaMemcpyAsync(&info, L.info, sizeof(info), cudaMemcpyDeviceToHost, s), "p2p_plan_create");
    FAIL_CUDA(cudaStreamSynchronize(s), "p2p_plan_create");
    if (info.status) {
        free(p);
        return P2P_ERR_INVALID;
    }
    int which = 0;
    if (choose) {
        // When most source lists hold just over one default chunk (193 .. 256 sources), every box would get a
        // full item and a short tail item with the same fixed cost; 256-source items (6 warps per block, so two
        // blocks still fit an SM) give those boxes one item each.  When the whole plan has fewer than 2.5 items
        // per resident warp (16 per SM), the last items of the heaviest-first list leave most warps idle;
        // 128-source items spread it (measured on the 32 768-point cube, 8^3 boxes: 3 584 items of 192
        // sources 60.4 us, 5 400 of 128 51.2 us, of 96 52.2 us, of 64 59.4 us).  The workspace is sized for
        // the narrow chunk.
        if (2ll * info.tails > nb) which = 1;
        else if (2ll * info.items[0] < 5ll * 16 * sms) which = 2;
        t.chunk = candidates[which]->chunk;
        t.warps_per_cta = candidates[which]->warps_per_cta;
        p->tune = t;
    }
    const int64_t items = info.items[which];
    k_list_sizes<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(L.list_len, nb, t.chunk, L.n_chunks, L.padded);
    FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/sizes");
    FAIL_CUDA(scan_exclusive_i32(L.n_chunks, L.item_off, nb, nullptr, L.scan_ws, s), "p2p_plan_create/scan");
    FAIL_CUDA(scan_exclusive_i32(L.padded, p->pk_off, nb, p->pk_off + nb, L.scan_ws, s),
              "p2p_plan_create/scan_lists");
    k_pack<<<blocks_for((int64_t)nb * 32, kThreads), kThreads, 0, s>>>(
        p->xs_src, p->src_box_ptr, in.nbr_ptr, in.nbr_idx, p->nbr_self, p->pk_off, nb, upper, p->nb_src, p->pk_xyz);
    FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/pack");
    if (layout == P2P_LAYOUT_REPETITION) {
        // per-target records (L.padded is free once the list offsets are scanned)
        k_rep_count<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(in.box_ptr, p->box_src, nb, L.padded);
        FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/rep_count");
        FAIL_CUDA(scan_exclusive_i32(L.padded, p->rec_boff, nb, p->rec_boff + nb, L.scan_ws, s),
                  "p2p_plan_create/rep_scan");
        k_rep_fill<<<blocks_for((int64_t)nb * 32, kThreads), kThreads, 0, s>>>(
            p->xs, in.perm, in.box_ptr, p->box_src, p->pk_off, p->nb_src, p->rec_boff, nb, n, p->rec_off, p->rec_xyz,
            p->rec_src);
        FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/rep_fill");
    }
    // few items: an exact order keeps the last ones short (32 768-point cube, 5 574 items: 53.3 us, by 8 bits 53.9)
    const bool fine = items <= 16384;
    k_item_records<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(L.n_chunks, L.item_off, in.box_ptr, L.list_len,
                                                                 L.self_len, p->pk_off, nb, t.chunk, t.target_group,
                                                                 p->two_sets, fine, L.recs, L.keys, L.vals);
    FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/items");
    if (items > 0) {
        bool in_alt = false;
        FAIL_CUDA(radix_sort_pairs(L.keys, L.vals, L.keys_alt, L.vals_alt, items, fine ? kFineCostBits : kCostBits,
                                   L.radix_ws, L.radix_bytes, s, &in_alt),
                  "p2p_plan_create/sort");
        k_item_gather<<<blocks_for(items, kThreads), kThreads, 0, s>>>(L.recs, in_alt ? L.vals_alt : L.vals, items,
                                                                       p->items);
        FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/order");
    }
    if (p->tc_pack)  // n_chunks and padded are free once the items are built
        FAIL_CUDA(p2p_tc_build(p, L.n_chunks, L.padded, L.scan_ws, s), "p2p_plan_create/tc_lists");
    p->tcb_groups = 0;
    if (p->tcb_gstart && p->nbs > 0)
        FAIL_CUDA(p2p_tcb_build(p, L.n_chunks, L.scan_ws, s), "p2p_plan_create/tc_box_lists");
    // direct kernel: one item per target box (the item-sort scratch is free again)
    p->direct_k = 0;
    if (layout != P2P_LAYOUT_SYMMETRIC && layout != P2P_LAYOUT_REPETITION) {
        int32_t wb = t.warp_boxes;
        if (wb == 0) {
            wb = plan_warp_boxes(n, nb, in.sources, kernel, layout);
            if (wb != -1 && heaviest_decides(wb, info, nb, sms)) wb = -1;
        }
        p->tune.warp_boxes = wb;
        if (wb > 0) {
            p->direct_k = wb;
            k_direct_items<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(in.box_ptr, L.list_len, L.self_len, p->pk_off,
                                                                         nb, 32 / wb, L.recs, L.keys, L.vals);
            FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/direct_items");
            bool in_alt = false;
            FAIL_CUDA(radix_sort_pairs(L.keys, L.vals, L.keys_alt, L.vals_alt, nb, kFineCostBits, L.radix_ws, L.radix_bytes, s, &in_alt),
                      "p2p_plan_create/direct_sort");
            k_item_gather<<<blocks_for(nb, kThreads), kThreads, 0, s>>>(L.recs, in_alt ? L.vals_alt : L.vals, nb,
                                                                        p->ditems);
            FAIL_CUDA(cudaGetLastError(), "p2p_plan_create/direct_order");
        }
    } else {
        p->tune.warp_boxes = -1;
    }
    // box-group kernel (indexed layout): groups of consecutive target boxes staging the union of their
    // neighbourhoods; a plan whose largest union does not fit the kernel's buffer keeps the staged pipeline
    p->group_k = 0;
    p->n_groups = 0;
    p->group_cap = 0;
    p->group_pos_cap = 0;
    p->group_asked = t.warp_boxes == -2;
    p->pairs = (int64_t)info.pairs;
    p->heavy = (int64_t)info.heavy;
    p->even = p->pairs / (32ll * sms);
    if (p->tune.warp_boxes == -2 && (layout != P2P_LAYOUT_INDEXED || nb == 0)) p->tune.warp_boxes = -1;
    int32_t cap[2] = {0, 0};
    if (p->tune.warp_boxes == -2) {
        p->n_groups = (nb + kGroupBoxes - 1) / kGroupBoxes;
        FAIL_CUDA(p2p_group_build(p, in.nbr_ptr, in.nbr_idx, L.keys, L.vals, L.keys_alt, L.vals_alt, L.radix_ws,
                                  L.radix_bytes, L.maxes, s, cap),
                  "p2p_plan_create/groups");
    }
    if (p->tcb_gstart && p->nbs > 0)
        FAIL_CUDA(cudaMemcpyAsync(&p->tcb_groups, p->tcb_gstart + p->nbs, sizeof(int32_t), cudaMemcpyDeviceToHost, s),
                  "p2p_plan_create/tc_box_groups");
    // the plan is complete when this returns: later calls may use it on any stream
    FAIL_CUDA(cudaStreamSynchronize(s), "p2p_plan_create");
    if (p->tune.warp_boxes == -2) {
        if (cap[0] > 0 && cap[0] <= kGroupCapMax) {
            p->group_k = 1;
            p->group_cap = (cap[0] + 3) & ~3;
            p->group_pos_cap = cap[1];
        } else {
            p->tune.warp_boxes = -1;
        }
    }
    p->max_chunks = (int32_t)(((int64_t)info.max_len + t.chunk - 1) / t.chunk);
    p->max_box = info.max_box;
    p->n_items = items;
    p->packed = info.packed;
    FAIL_CUDA(p2p_pair_configure(p), "p2p_plan_create/occupancy");
    // a second or third wave of two blocks per SM that runs partly empty, on a surface: the staged pipeline
    // (auto_warp_boxes, D = 20 - 23)
    if (t.warp_boxes == 0 && p->group_k && n > 20ll * nb && in.sources <= 300ll * nb && p->group_grid <= 2 * sms &&
        p->n_groups > p->group_grid && 2 * p->n_groups <= 5 * p->group_grid) {
        p->group_k = 0;
        p->tune.warp_boxes = -1;
    }
#undef FAIL_CUDA
    *plan = p;
    return P2P_OK;
}

}  // namespace

extern "C" {

P2P_API p2p_status p2p_build_neighbors(const int64_t* box_keys, const int32_t* box_ptr, int32_t num_boxes,
                                       int32_t ng, int32_t* nbr_ptr, int32_t* nbr_idx, int64_t* nnz,
                                       int64_t* sources, void* work, size_t work_bytes, p2p_stream_t stream) {
    return build_neighbors(box_keys, num_boxes, box_keys, box_ptr, num_boxes, ng, nbr_ptr, nbr_idx, nullptr, nnz,
                           sources, work, work_bytes, (cudaStream_t)stream, false);
}

P2P_API p2p_status p2p_build_neighbors_st(const int64_t* tgt_keys, int32_t num_tgt_boxes, const int64_t* src_keys,
                                          const int32_t* src_box_ptr, int32_t num_src_boxes, int32_t ng,
                                          int32_t* nbr_ptr, int32_t* nbr_idx, int32_t* nbr_self, int64_t* nnz,
                                          int64_t* sources, void* work, size_t work_bytes, p2p_stream_t stream) {
    if (num_src_boxes == 0 && num_tgt_boxes > 0) {
        // no sources: every list is empty
        if (!nbr_ptr || !nbr_self || !nnz || !sources) return P2P_ERR_INVALID;
        cudaStream_t s = (cudaStream_t)stream;
        *nnz = 0;
        *sources = 0;
        P2P_TRY_CUDA(cudaMemsetAsync(nbr_ptr, 0, sizeof(int32_t) * ((size_t)num_tgt_boxes + 1), s),
                     "p2p_build_neighbors_st");
        P2P_TRY_CUDA(cudaMemsetAsync(nbr_self, 0xff, sizeof(int32_t) * (size_t)num_tgt_boxes, s),
                     "p2p_build_neighbors_st");
        P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_build_neighbors_st");
        return P2P_OK;
    }
    return build_neighbors(tgt_keys, num_tgt_boxes, src_keys, src_box_ptr, num_src_boxes, ng, nbr_ptr, nbr_idx,
                           nbr_self, nnz, sources, work, work_bytes, (cudaStream_t)stream, true);
}

P2P_API p2p_status p2p_plan_workspace_size(int64_t n, int32_t num_boxes, int64_t nnz, int64_t sources,
                                           p2p_layout layout, int32_t max_nrhs, const p2p_tuning* tuning,
                                           size_t* bytes) {
    if (!bytes) return P2P_ERR_INVALID;
    if (layout == P2P_LAYOUT_REPETITION) return P2P_ERR_INVALID;  // its records: p2p_plan_workspace_size_rep
    p2p_status st = check_sizes(n, num_boxes, n, num_boxes, sources, layout, max_nrhs, false);
    if (st != P2P_OK) return st;
    p2p_tuning t = resolve_tuning(tuning);
    if (!tuning_valid(t)) return P2P_ERR_INVALID;
    *bytes = plan_layout(n, num_boxes, n, num_boxes, false, sources, nnz, layout, max_nrhs, t, nullptr).bytes;
    return P2P_OK;
}

P2P_API p2p_status p2p_repetition_records(const int32_t* box_ptr, int32_t num_boxes, const int32_t* nbr_ptr,
                                          const int32_t* nbr_idx, int64_t* records, p2p_stream_t stream) {
    if (!records || num_boxes < 0 || (num_boxes > 0 && (!box_ptr || !nbr_ptr || !nbr_idx))) return P2P_ERR_INVALID;
    return repetition_records(box_ptr, num_boxes, nbr_ptr, nbr_idx, records, (cudaStream_t)stream);
}

P2P_API p2p_status p2p_plan_workspace_size_rep(int64_t n, int32_t num_boxes, int64_t nnz, int64_t sources,
                                               int64_t records, const p2p_tuning* tuning, size_t* bytes) {
    if (!bytes || records < 0 || records >= INT32_MAX) return P2P_ERR_INVALID;
    p2p_status st = check_sizes(n, num_boxes, n, num_boxes, sources, P2P_LAYOUT_REPETITION, 1, false);
    if (st != P2P_OK) return st;
    p2p_tuning t = resolve_tuning(tuning);
    if (!tuning_valid(t)) return P2P_ERR_INVALID;
    *bytes = plan_layout(n, num_boxes, n, num_boxes, false, sources, nnz, P2P_LAYOUT_REPETITION, 1, t, nullptr, records)
                 .bytes;
    return P2P_OK;
}

P2P_API p2p_status p2p_plan_workspace_size_st(int64_t n_tgt, int32_t num_tgt_boxes, int64_t n_src,
                                              int32_t num_src_boxes, int64_t nnz, int64_t sources, p2p_layout layout,
                                              int32_t max_nrhs, const p2p_tuning* tuning, size_t* bytes) {
    if (!bytes) return P2P_ERR_INVALID;
    p2p_status st = check_sizes(n_tgt, num_tgt_boxes, n_src, num_src_boxes, sources, layout, max_nrhs, true);
    if (st != P2P_OK) return st;
    p2p_tuning t = resolve_tuning(tuning);
    if (!tuning_valid(t)) return P2P_ERR_INVALID;
    *bytes = plan_layout(n_tgt, num_tgt_boxes, n_src, num_src_boxes, true, sources, nnz, layout, max_nrhs, t, nullptr)
                 .bytes;
    return P2P_OK;
}

P2P_API p2p_status p2p_plan_create(p2p_plan** plan, const float* pts, int64_t n, const int32_t* perm,
                                   const int32_t* box_ptr, int32_t num_boxes, const int32_t* nbr_ptr,
                                   const int32_t* nbr_idx, int64_t nnz, int64_t sources, p2p_kernel kernel, float k,
                                   p2p_layout layout, int32_t max_nrhs, const p2p_tuning* tuning, void* workspace,
                                   size_t workspace_bytes, p2p_stream_t stream) {
    PlanInput in{pts, n, perm, box_ptr, num_boxes, pts, n, perm, box_ptr, num_boxes, nbr_ptr, nbr_idx, nullptr,
                 nnz, sources, false};
    return plan_create(plan, in, kernel, k, layout, max_nrhs, tuning, workspace, workspace_bytes,
                       (cudaStream_t)stream);
}

P2P_API p2p_status p2p_plan_create_st(p2p_plan** plan, const float* tgt_pts, int64_t n_tgt, const int32_t* tgt_perm,
                                      const int32_t* tgt_box_ptr, int32_t num_tgt_boxes, const float* src_pts,
                                      int64_t n_src, const int32_t* src_perm, const int32_t* src_box_ptr,
                                      int32_t num_src_boxes, const int32_t* nbr_ptr, const int32_t* nbr_idx,
                                      const int32_t* nbr_self, int64_t nnz, int64_t sources, p2p_kernel kernel,
                                      float k, p2p_layout layout, int32_t max_nrhs, const p2p_tuning* tuning,
                                      void* workspace, size_t workspace_bytes, p2p_stream_t stream) {
    PlanInput in{tgt_pts, n_tgt, tgt_perm, tgt_box_ptr, num_tgt_boxes, src_pts, n_src, src_perm, src_box_ptr,
                 num_src_boxes, nbr_ptr, nbr_idx, nbr_self, nnz, sources, true};
    return plan_create(plan, in, kernel, k, layout, max_nrhs, tuning, workspace, workspace_bytes,
                       (cudaStream_t)stream);
}

P2P_API p2p_status p2p_plan_destroy(p2p_plan* plan) {
    free(plan);
    return P2P_OK;
}

P2P_API p2p_status p2p_plan_info(const p2p_plan* plan, int64_t* n, int32_t* num_boxes, int64_t* sources,
                                 int64_t* work_items, p2p_layout* layout, p2p_tuning* tuning) {
    if (!plan) return P2P_ERR_INVALID;
    if (n) *n = plan->n;
    if (num_boxes) *num_boxes = plan->nb;
    if (sources) *sources = plan->sources;
    if (work_items) *work_items = plan->n_items;
    if (layout) *layout = plan->layout;
    if (tuning) *tuning = plan->tune;
    return P2P_OK;
}

P2P_API p2p_status p2p_plan_pair_count(const p2p_plan* plan, int64_t* pairs, p2p_stream_t stream) {
    if (!plan || !pairs) return P2P_ERR_INVALID;
    *pairs = 0;
    if (plan->n == 0) return P2P_OK;
    cudaStream_t s = (cudaStream_t)stream;
    P2P_TRY_CUDA(cudaMemsetAsync(plan->scratch64, 0, sizeof(long long), s), "p2p_plan_pair_count");
    k_pair_count<<<blocks_for((int64_t)plan->nb * 32, kThreads), kThreads, 0, s>>>(
        plan->xs, plan->box_ptr, plan->xs_src, plan->src_box_ptr, plan->nbr_ptr, plan->nbr_idx, plan->nbr_self,
        plan->box_src, plan->nb, (unsigned long long*)plan->scratch64);
    P2P_CHECK_LAUNCH("p2p_plan_pair_count");
    long long v = 0;
    P2P_TRY_CUDA(cudaMemcpyAsync(&v, plan->scratch64, sizeof(v), cudaMemcpyDeviceToHost, s), "p2p_plan_pair_count");
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_plan_pair_count");
    *pairs = v;
    return P2P_OK;
}

P2P_API p2p_status p2p_plan_update_points(p2p_plan* plan, const float* pts, const double lo[3], double h, int32_t ng,
                                          int64_t* moved, p2p_stream_t stream) {
    if (moved) *moved = 0;
    if (!plan || !lo || !(h > 0.0) || !isfinite(h) || ng < 1 || ng > (1 << 21)) return P2P_ERR_INVALID;
    if (!isfinite(lo[0]) || !isfinite(lo[1]) || !isfinite(lo[2])) return P2P_ERR_INVALID;
    if (plan->two_sets) return P2P_ERR_UNSUPPORTED;
    if (plan->n == 0) return P2P_OK;
    if (!pts || ((uintptr_t)pts & 3)) return P2P_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    // scratch64[0]: moved count, scratch64[1]: non-finite flag (the pair count's slot, free between calls)
    P2P_TRY_CUDA(cudaMemsetAsync(plan->scratch64, 0, 2 * sizeof(long long), s), "p2p_plan_update_points");
    k_moved<<<blocks_for(plan->n, kThreads), kThreads, 0, s>>>(pts, plan->perm, plan->xs, plan->n, lo[0], lo[1], lo[2],
                                                               h, ng, (unsigned long long*)plan->scratch64,
                                                               (int32_t*)(plan->scratch64 + 1));
    P2P_CHECK_LAUNCH("p2p_plan_update_points/check");
    long long host[2] = {0, 0};
    P2P_TRY_CUDA(cudaMemcpyAsync(host, plan->scratch64, sizeof(host), cudaMemcpyDeviceToHost, s),
                 "p2p_plan_update_points");
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_plan_update_points");
    if (host[1]) return P2P_ERR_INVALID;
    if (moved) *moved = host[0];
    if (host[0]) return P2P_ERR_STALE;
    k_gather_xyz<<<blocks_for(plan->n, kThreads), kThreads, 0, s>>>(pts, plan->perm, plan->n, plan->xs);
    P2P_CHECK_LAUNCH("p2p_plan_update_points/gather");
    if (plan->pk_xyz && plan->packed > 0) {
        k_repack_xyz<<<blocks_for(plan->packed, kThreads), kThreads, 0, s>>>(plan->xs, plan->nb_src, plan->packed,
                                                                             plan->pk_xyz);
        P2P_CHECK_LAUNCH("p2p_plan_update_points/repack");
    }
    plan->pts = pts;
    plan->src_pts = pts;
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_plan_update_points");
    return P2P_OK;
}

P2P_API p2p_status p2p_last_async_status(const p2p_plan* plan, p2p_stream_t stream) {
    if (!plan) return P2P_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned int v = 0;
    P2P_TRY_CUDA(cudaMemcpyAsync(&v, plan->status, sizeof(v), cudaMemcpyDeviceToHost, s), "p2p_last_async_status");
    P2P_TRY_CUDA(cudaMemsetAsync(plan->status, 0, sizeof(unsigned int), s), "p2p_last_async_status");
    P2P_TRY_CUDA(cudaStreamSynchronize(s), "p2p_last_async_status");
    if (v & P2P_DEV_TIMEOUT) return P2P_ERR_TIMEOUT;
    if (v & P2P_DEV_BAD_INPUT) return P2P_ERR_INVALID;
    if (v & P2P_DEV_TC_FAULTED) return P2P_ERR_UNSUPPORTED;
    return P2P_OK;
}

}  // extern "C"
