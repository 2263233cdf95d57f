// Apply path of the P2P operator: strength staging (the gather into box-sorted
// order, the repack into the repetition layout's records), the FP32 pair kernel, its adjoint and the coordinate gradient.
//
// The pair kernel's device code (work items, staging, lane mapping) lives in
// p2p_pair.cuh, shared with the persistent batched launch.
#include <math.h>

#include <algorithm>

#include "p2p_direct.cuh"
#include "p2p_pair.cuh"

using namespace p2p_detail;
using namespace p2p_pair;
using p2p_direct::DirectArgs;
using p2p_direct::kDirectWarps;

namespace {

// Persistent pair kernel: the warps of the grid take turns in the plan's heaviest-first item list.
template <int R>
__global__ void __launch_bounds__(P2P_PAIR_MAX_THREADS, R == 1 ? P2P_PAIR_MIN_BLOCKS : 1)
    k_pair(const __grid_constant__ PairArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int warps = blockDim.x >> 5;
    unsigned char* ws = smem_raw + (size_t)warp * warp_smem_bytes(a.chunk, R, a.sym);
    run_pipeline<R>(ws, a.chunk, a.sym != 0, lane, true, a.items, a.n_items, (int64_t)blockIdx.x * warps + warp,
                    (int64_t)gridDim.x * warps, a.status, [&](const ItemRec&) -> const PairArgs* { return &a; });
}

// Direct kernel (sparse boxes, one right-hand side): warp w of the persistent
// grid serves K boxes at a time, sources read through the L1 (p2p_direct.cuh).
#ifndef P2P_DIRECT_MIN_BLOCKS
#define P2P_DIRECT_MIN_BLOCKS 4
#endif
template <int KERN, bool RED, int K>
__global__ void __launch_bounds__(kDirectWarps * 32, P2P_DIRECT_MIN_BLOCKS)
    k_pair_direct(const __grid_constant__ DirectArgs a) {
    __shared__ float2 red[kDirectWarps][4 * 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    p2p_direct::run_direct<KERN, RED, K>(a, red[warp], (int)blockIdx.x * kDirectWarps + warp,
                                         (int64_t)gridDim.x * kDirectWarps, lane);
}

using DirectKernel = void (*)(DirectArgs);

// Repetition layout (Sec. 3.3, eq. 9): one thread per target, reading its own record front to back -- entry 0
// its coordinates, entries 1 .. S_b its neighbourhood's sources with the strengths repacked at this apply.  The
// record holds the target itself among its own box's sources: the r = 0 mask applies to every entry.
template <int KERN>
__global__ void __launch_bounds__(256) k_pair_rep(const int32_t* __restrict__ rec_off,
                                                  const float4* __restrict__ rec_xyz,
                                                  const float2* __restrict__ rec_lam, const int32_t* __restrict__ perm,
                                                  int64_t n, float k, float2* __restrict__ out, int64_t ld) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int32_t off = rec_off[t], end = rec_off[t + 1];
    const float4 x = rec_xyz[off];
    const float4 tx[1] = {x};
    float2 acc[1][1] = {{make_float2(0.f, 0.f)}};
    for (int32_t e = off + 1; e < end; ++e) {
        const float2 l[1] = {rec_lam[e]};
        pair_core<KERN, 1, 1, true>(rec_xyz[e], l, tx, acc, k);
    }
    out[(int64_t)perm[t] * ld] = make_float2(acc[0][0].x * kInv4Pi, acc[0][0].y * kInv4Pi);
}

template <int KERN, bool RED>
DirectKernel direct_kernel_k(int k) {
    switch (k) {
        case 1: return k_pair_direct<KERN, RED, 1>;
        case 2: return k_pair_direct<KERN, RED, 2>;
        case 4: return k_pair_direct<KERN, RED, 4>;
        case 8: return k_pair_direct<KERN, RED, 8>;
        case 16: return k_pair_direct<KERN, RED, 16>;
        default: return k_pair_direct<KERN, RED, 32>;
    }
}

DirectKernel direct_kernel(const p2p_plan* p) {
    const bool red = p->layout == P2P_LAYOUT_REDUNDANT;
    if (p->kernel == P2P_HELMHOLTZ)
        return red ? direct_kernel_k<P2P_HELMHOLTZ, true>(p->direct_k) : direct_kernel_k<P2P_HELMHOLTZ, false>(p->direct_k);
    return red ? direct_kernel_k<P2P_LAPLACE, true>(p->direct_k) : direct_kernel_k<P2P_LAPLACE, false>(p->direct_k);
}

// ----------------------------------------------------------------- staging --

// dst[s * nrhs + q] = src[rows[s] * ld + q]  (rows[s] < 0: zero)
__global__ void k_gather_rows(const float2* __restrict__ src, int64_t ld, const int32_t* __restrict__ rows, int64_t n,
                              int32_t nrhs, float2* __restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * nrhs) return;
    const int64_t s = i / nrhs;
    const int q = (int)(i - s * nrhs);
    const int32_t r = rows[s];
    dst[i] = r >= 0 ? src[(int64_t)r * ld + q] : make_float2(0.f, 0.f);
}

// One right-hand side, four rows per thread: dst[s] = src[rows[s] * ld]
// (rows[s] < 0: zero) with a 16-byte index load, four independent gathers
// and two 16-byte stores.  rows and dst are 16-byte aligned.
__global__ void k_gather_rows4(const float2* __restrict__ src, int64_t ld, const int32_t* __restrict__ rows, int64_t n,
                               float2* __restrict__ dst) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t s0 = q * 4;
    if (s0 >= n) return;
    if (s0 + 4 <= n) {
        const int4 r = *reinterpret_cast<const int4*>(rows + s0);
        const float2 z = make_float2(0.f, 0.f);
        const float2 v0 = r.x >= 0 ? src[(int64_t)r.x * ld] : z;
        const float2 v1 = r.y >= 0 ? src[(int64_t)r.y * ld] : z;
        const float2 v2 = r.z >= 0 ? src[(int64_t)r.z * ld] : z;
        const float2 v3 = r.w >= 0 ? src[(int64_t)r.w * ld] : z;
        reinterpret_cast<float4*>(dst + s0)[0] = make_float4(v0.x, v0.y, v1.x, v1.y);
        reinterpret_cast<float4*>(dst + s0)[1] = make_float4(v2.x, v2.y, v3.x, v3.y);
    } else {
        for (int64_t s = s0; s < n; ++s) dst[s] = rows[s] >= 0 ? src[(int64_t)rows[s] * ld] : make_float2(0.f, 0.f);
    }
}

cudaError_t stage_rows(const float2* src, int64_t ld, const int32_t* rows, int64_t nrows, int32_t nrhs, float2* dst,
                       cudaStream_t s) {
    if (nrows <= 0) return cudaSuccess;
    if (nrhs == 1) {
        const int64_t threads = (nrows + 3) / 4;
        k_gather_rows4<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(src, ld, rows, nrows, dst);
    } else {
        const int64_t total = nrows * nrhs;
        k_gather_rows<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(src, ld, rows, nrows, nrhs, dst);
    }
    return cudaGetLastError();
}

// dst[s * nrhs + q] = (|src[rows[s] * ld + q]|, 0)  (rows[s] < 0: zero): the strengths' magnitudes, for the sums
// of the terms' magnitudes of a guarded apply.
__global__ void k_gather_abs(const float2* __restrict__ src, int64_t ld, const int32_t* __restrict__ rows, int64_t n,
                             int32_t nrhs, float2* __restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * nrhs) return;
    const int64_t s = i / nrhs;
    const int q = (int)(i - s * nrhs);
    const int32_t r = rows[s];
    float m = 0.f;
    if (r >= 0) {
        const float2 v = src[(int64_t)r * ld + q];
        m = hypotf(v.x, v.y);
    }
    dst[i] = make_float2(m, 0.f);
}

int r_index(int R) { return R == 1 ? 0 : (R == 2 ? 1 : 2); }

// The dynamic shared-memory limit is an attribute of the kernel function,
// shared by every plan: it only ever grows (to the largest launch seen), so no
// plan's configuration can lower it below another plan's launch.
int g_smem_attr[3] = {0, 0, 0};

template <int R>
cudaError_t raise_smem_limit(int smem) {
    int& cur = g_smem_attr[r_index(R)];
    if (smem <= __atomic_load_n(&cur, __ATOMIC_ACQUIRE)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_pair<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) {
        int seen = __atomic_load_n(&cur, __ATOMIC_ACQUIRE);
        while (seen < smem && !__atomic_compare_exchange_n(&cur, &seen, smem, false, __ATOMIC_ACQ_REL, __ATOMIC_ACQUIRE)) {
        }
    }
    return e;
}

template <int R>
cudaError_t configure_r(p2p_plan* p) {
    const int ri = r_index(R);
    p->grid[ri] = 0;
    p->grid_warps[ri] = 0;
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k_pair<R>);
    if (e != cudaSuccess) return e;
    const bool sym = p->layout == P2P_LAYOUT_SYMMETRIC;
    // the tuning's warps per block, halved until one block fits (threads, shared memory)
    for (int warps = p->tune.warps_per_cta; warps >= 1; warps >>= 1) {
        const int smem = warps * warp_smem_bytes(p->tune.chunk, R, sym);
        if (smem > optin || warps * 32 > fa.maxThreadsPerBlock) continue;
        e = raise_smem_limit<R>(smem);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pair<R>, warps * 32, smem);
        if (e != cudaSuccess) return e;
        if (per_sm > 0) {
            p->grid[ri] = per_sm * sms;
            p->grid_warps[ri] = warps;
            return cudaSuccess;
        }
    }
    return cudaSuccess;  // no block fits: the launch reports P2P_ERR_UNSUPPORTED
}

template <int R>
p2p_status launch_pair(const p2p_plan* p, const PairArgs& a, cudaStream_t s) {
    const int warps = p->grid_warps[r_index(R)];
    const int smem = warps * warp_smem_bytes(a.chunk, R, a.sym != 0);
    int grid = p->grid[r_index(R)];
    if (grid <= 0) {
        set_message("p2p_apply: the pair kernel does not fit on this device with this tuning (shared memory)");
        return P2P_ERR_UNSUPPORTED;
    }
    if ((int64_t)grid * warps > a.n_items) grid = (int)((a.n_items + warps - 1) / warps);
    P2P_TRY_CUDA(raise_smem_limit<R>(smem), "p2p_apply/attribute");
    k_pair<R><<<grid, warps * 32, smem, s>>>(a);
    P2P_CHECK_LAUNCH("p2p_apply/pair");
    return P2P_OK;
}

// lam: strengths (one row per source, may be NULL when there are none); out: results (one row per target).
p2p_status check_apply_args(const p2p_plan* plan, const void* lam, const void* out, int32_t nrhs, int64_t ld) {
    if (!plan || nrhs < 1 || nrhs > plan->max_nrhs || ld < nrhs) return P2P_ERR_INVALID;
    if ((plan->n_src > 0 && !lam) || (plan->n > 0 && !out)) return P2P_ERR_INVALID;
    if (((uintptr_t)lam & 7) || ((uintptr_t)out & 7)) return P2P_ERR_INVALID;
    return P2P_OK;
}

}  // namespace

// S[perm[t] * nrhs + q] = sum over the sources s of target t's neighbourhood (r > 0) of |lambda_sq| / (4 pi r),
// i.e. sum_s |G(r) lambda_sq| for both kernels (|exp(ikr)| = 1), through the staged pipeline with the Laplace
// kernel on the strengths' magnitudes (lambda: leading dimension ld; S: nrhs).  Uses the plan's staging buffer.
p2p_status p2p_abs_sums(const p2p_plan* plan, const float2* lam, int64_t ld, int32_t nrhs, float2* S, cudaStream_t s) {
    const int32_t* rows = plan->src_perm;
    const int64_t nrows = plan->n_src;
    if (nrows > 0) {
        const int64_t total = nrows * nrhs;
        k_gather_abs<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(lam, ld, rows, nrows, nrhs, plan->lam_buf);
        P2P_CHECK_LAUNCH("p2p_apply_guarded/abs");
    }
    P2P_TRY_CUDA(cudaMemsetAsync(S, 0, (size_t)plan->n * nrhs * 8, s), "p2p_apply_guarded");
    if (plan->n_items == 0 || nrows == 0) return P2P_OK;
    PairArgs a = base_args(plan);
    a.out = S;
    a.ld = nrhs;
    a.nrhs = nrhs;
    a.kernel = P2P_LAPLACE;
    a.k = 0.f;
    a.atomic_out = 1;  // the buffer is zeroed above
    const int R = nrhs >= 4 ? 4 : (nrhs >= 2 ? 2 : 1);
    return R == 1 ? launch_pair<1>(plan, a, s) : (R == 2 ? launch_pair<2>(plan, a, s) : launch_pair<4>(plan, a, s));
}

cudaError_t p2p_group_configure(p2p_plan* p);
cudaError_t p2p_multi_configure(p2p_plan* p);
p2p_status p2p_multi_stage(const p2p_plan* p, const float2* lam, int32_t nrhs, int64_t ld, cudaStream_t s);
p2p_status p2p_multi_launch(const p2p_plan* p, float2* out, int32_t nrhs, int64_t ld, float k, cudaStream_t s);
p2p_status p2p_grad_launch(const p2p_plan* p, const float2* lam, const float2* g, float* grad, int32_t nrhs, int64_t ld,
                           cudaStream_t s);
p2p_status p2p_group_launch(const p2p_plan* p, float2* out, int64_t ld, float k, cudaStream_t s);

cudaError_t p2p_pair_configure(p2p_plan* plan) {
    cudaError_t e = p2p_group_configure(plan);
    if (e == cudaSuccess && plan->max_nrhs > 1) e = p2p_multi_configure(plan);
    if (e == cudaSuccess) e = configure_r<1>(plan);
    if (e == cudaSuccess && plan->max_nrhs >= 2) e = configure_r<2>(plan);
    if (e == cudaSuccess && plan->max_nrhs >= 4) e = configure_r<4>(plan);
    plan->direct_grid = 0;
    if (e == cudaSuccess && plan->direct_k > 0) {
        int dev = 0, sms = 0, per_sm = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, direct_kernel(plan), kDirectWarps * 32, 0);
        if (e == cudaSuccess) plan->direct_grid = per_sm * sms;
    }
    return e;
}

// Entries shared with the tensor-core translation unit.
p2p_status p2p_tc_stage(const p2p_plan* plan, const float2* lam, int32_t nrhs, int64_t ld, int np,
                        cudaStream_t s);
p2p_status p2p_apply_tc(const p2p_plan* plan, float2* out, int32_t nrhs, int64_t ld, int32_t adjoint, int np,
                        cudaStream_t s);
bool p2p_tc_supported(const p2p_plan* plan, int32_t nrhs);
p2p_status p2p_tcb_stage(const p2p_plan* plan, const float2* lam, int32_t nrhs, int64_t ld, int np, cudaStream_t s);
p2p_status p2p_tcb_apply(const p2p_plan* plan, float2* out, int32_t nrhs, int64_t ld, int32_t adjoint, int np,
                         cudaStream_t s);

extern "C" {

static p2p_path resolve_path(const p2p_plan* plan, int32_t nrhs, p2p_path path) {
    if (path == P2P_PATH_AUTO)
        return (nrhs >= 16 && p2p_tc_supported(plan, nrhs)) ? P2P_PATH_TC_BF16X3 : P2P_PATH_FP32_SHARED;
    return path;
}

static bool is_tc(p2p_path path) { return path == P2P_PATH_TC_BF16X3 || path == P2P_PATH_TC_BF16X6; }
// Several right-hand sides on the streamed kernel (p2p_multi.cu): every layout with full source lists, from the sorted
// strengths.  Two of them stay with the staged pipeline where one box's chain decides, since the streamed kernel stages a
// box's list once per 32 targets: where the plan has few boxes, fewer the more points each holds, and where its heaviest
// box is worth more than twenty average warps.  Measured with two right-hand sides, streamed / staged, us, on
// spheres: 1132 boxes of 7 points 19.5 / 19.5, 2326 of 7 21 / 21, 3850 of 7 23 / 25; 499 of 16 30 / 27, 2672 of 16 35 / 40;
// 620 of 26 30 / 28, 2279 of 29 (Laplace) 43 / 38, 4191 of 29 80 / 92 (Laplace 62 / 69); 1389 of 47 71 / 64 (Laplace 54 / 46),
// 7156 of 42 233 / 249; on clustered assemblies by heaviest box / average warp: 30 - 40 (70 001 points at 9 to 12 per box)
// 64 / 57 and 74 / 65 (Laplace 50 / 42 and 58 / 48), 25 (100 001) 75 / 77 and 98 / 94 (59 / 57, 73 / 64), 10 (400 001) 188 / 220
// and 243 / 263 (139 / 159).  From three right-hand sides on the streamed kernel won everywhere from 8 000 points up (499
// boxes of 16 with three: 34 / 42).
static bool is_multi(const p2p_plan* plan, int32_t nrhs, p2p_path path) {
    if (path != P2P_PATH_FP32_SHARED || nrhs < 2) return false;
    if (plan->layout != P2P_LAYOUT_INDEXED && plan->layout != P2P_LAYOUT_REDUNDANT) return false;
    return nrhs > 2 || (plan->nb >= 2048 && (int64_t)plan->nb * plan->nb >= 80 * plan->n && plan->heavy <= 20 * plan->even);
}
static int tc_parts(p2p_path path) { return path == P2P_PATH_TC_BF16X6 ? 3 : 2; }
// One box per unit (p2p_tc_box.cu) instead of 128 targets: where units of 128 targets are too few for the SMs, and for
// three parts with more than 32 right-hand sides per launch, whose chains would have to be too short (kSegment).  With long
// lists and the Helmholtz kernel, where a unit takes longest, a second or third round of the SMs that is nearly empty (152
// units are 19 456 targets) costs more than it does elsewhere, so the lines lie a little higher.
// Measured on spheres at 20 points per box, us, 128 targets / one box: hi / lo, 16 right-hand sides, 8 193 points 48 / 39,
// 16 385 62 / 55, 30 001 73 / 93; 64: 16 385 69 / 56, 30 001 89 / 93 (at 45 per box 117 / 111), 60 001 141 / 157; three
// parts, 32: 8 193 66 / 52, 16 385 76 / 77, 30 001 99 / 124; 64: 60 001 260 / 227.  Long lists, Helmholtz: ellipsoid at 48 per
// box, 24: 20 001 88 / 77, three parts 12 501 94 / 85; cube at 24 per box, 24: 20 001 95 / 92, 26 001 103 / 96, 33 001 level; 64:
// 41 001 163 / 138, 47 001 172 / 158, 52 001 level; three parts, 24: 16 001 95 / 86, 20 001 level (at 48 per box 21 501 147 / 137).
static bool tc_by_box(const p2p_plan* plan, int32_t nrhs, int parts) {
    if (!plan->tcb_gstart) return false;
    const bool wide = p2p_tc_launch_rhs(nrhs) > 32;
    if (parts == 3 && wide) return true;
    const bool dense = plan->kernel == P2P_HELMHOLTZ && plan->sources >= 240ll * plan->nb;
    const bool volume = plan->sources > 16ll * plan->n;  // 9 - 15 sources per target and point of a box on a surface
    int64_t limit = parts == 3 ? 12000 : (wide ? kTcBoxTargets : 20000);
    if (dense) limit = parts == 3 ? (volume ? 22000 : 14000) : (wide ? (volume ? 50000 : limit) : (volume ? 30000 : 22000));
    return plan->n < limit;
}

P2P_API p2p_status p2p_apply_stage(const p2p_plan* plan, const void* lambda, int32_t nrhs, int64_t ld, p2p_path path,
                                   p2p_stream_t stream) {
    if (!plan) return P2P_ERR_INVALID;
    p2p_status st = check_apply_args(plan, lambda, plan->n > 0 ? plan : nullptr, nrhs, ld);
    if (st != P2P_OK) return st;
    if (path < P2P_PATH_AUTO || path > P2P_PATH_TC_BF16X6) return P2P_ERR_INVALID;
    if (plan->n == 0 || plan->n_src == 0) return P2P_OK;
    path = resolve_path(plan, nrhs, path);
    if (is_tc(path) && !p2p_tc_supported(plan, nrhs)) return P2P_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    if (is_tc(path))
        return (tc_by_box(plan, nrhs, tc_parts(path)) ? p2p_tcb_stage : p2p_tc_stage)(plan, (const float2*)lambda, nrhs, ld,
                                                                                       tc_parts(path), s);
    if (is_multi(plan, nrhs, path)) return p2p_multi_stage(plan, (const float2*)lambda, nrhs, ld, s);
    if (plan->layout == P2P_LAYOUT_REPETITION) {
        // every target's record gets its own copy of its sources' strengths (the record head: 0)
        P2P_TRY_CUDA(stage_rows((const float2*)lambda, ld, plan->rec_src, plan->records, 1, plan->lam_buf, s),
                     "p2p_apply_stage");
        return P2P_OK;
    }
    P2P_TRY_CUDA(stage_rows((const float2*)lambda, ld, plan->src_perm, plan->n_src, nrhs, plan->lam_buf, s),
                 "p2p_apply_stage");  // strengths live on the sources
    return P2P_OK;
}

P2P_API p2p_status p2p_apply_staged(const p2p_plan* plan, void* out, int32_t nrhs, int64_t ld, int32_t adjoint,
                                    p2p_path path, p2p_stream_t stream) {
    if (!plan) return P2P_ERR_INVALID;
    p2p_status st = check_apply_args(plan, plan->n_src > 0 ? plan : nullptr, out, nrhs, ld);
    if (st != P2P_OK) return st;
    if (path < P2P_PATH_AUTO || path > P2P_PATH_TC_BF16X6) return P2P_ERR_INVALID;
    if (plan->n == 0) return P2P_OK;
    path = resolve_path(plan, nrhs, path);
    if (is_tc(path) && !p2p_tc_supported(plan, nrhs)) return P2P_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    // a two-set plan may have target boxes without any source nearby: no item or unit writes their rows
    if (plan->two_sets)
        P2P_TRY_CUDA(cudaMemset2DAsync(out, (size_t)ld * 8, 0, (size_t)nrhs * 8, (size_t)plan->n, s), "p2p_apply/zero");
    if (plan->n_src == 0) return P2P_OK;
    if (is_tc(path))
        return (tc_by_box(plan, nrhs, tc_parts(path)) ? p2p_tcb_apply : p2p_apply_tc)(plan, (float2*)out, nrhs, ld, adjoint,
                                                                                      tc_parts(path), s);
    if (plan->layout == P2P_LAYOUT_REPETITION) {
        const float k = adjoint ? -plan->k : plan->k;
        const unsigned blocks = (unsigned)((plan->n + 255) / 256);
        if (plan->kernel == P2P_HELMHOLTZ)
            k_pair_rep<P2P_HELMHOLTZ><<<blocks, 256, 0, s>>>(plan->rec_off, plan->rec_xyz, plan->lam_buf, plan->perm,
                                                              plan->n, k, (float2*)out, ld);
        else
            k_pair_rep<P2P_LAPLACE><<<blocks, 256, 0, s>>>(plan->rec_off, plan->rec_xyz, plan->lam_buf, plan->perm,
                                                            plan->n, k, (float2*)out, ld);
        P2P_CHECK_LAUNCH("p2p_apply/repetition");
        return P2P_OK;
    }
    PairArgs a = base_args(plan);
    a.out = (float2*)out;
    a.ld = ld;
    a.nrhs = nrhs;
    if (adjoint) a.k = -a.k;
    if (nrhs == 1 && plan->group_k && plan->group_grid > 0) {
        // one right-hand side, groups of boxes staging the union of their neighbourhoods once
        return p2p_group_launch(plan, (float2*)out, ld, a.k, s);
    }
    if (nrhs == 1 && plan->direct_k > 0 && plan->direct_grid > 0) {
        // one right-hand side on sparse boxes: the direct kernel, one item per box, every row stored once
        DirectArgs d;
        d.items = plan->ditems;
        d.n_items = plan->nb;
        d.xs = plan->xs_src;
        d.xt = plan->xs;
        d.pk_xyz = plan->pk_xyz;
        d.nb_src = plan->nb_src;
        d.lam = plan->lam_buf;
        d.perm = plan->perm;
        d.out = (float2*)out;
        d.ld = ld;
        d.k = a.k;
        const int64_t blocks_needed = (plan->nb + (int64_t)kDirectWarps * plan->direct_k - 1) /
                                      ((int64_t)kDirectWarps * plan->direct_k);
        const int grid = (int)std::min<int64_t>(plan->direct_grid, blocks_needed);
        direct_kernel(plan)<<<grid, kDirectWarps * 32, 0, s>>>(d);
        P2P_CHECK_LAUNCH("p2p_apply/direct");
        return P2P_OK;
    }
    if (a.atomic_out && !plan->two_sets)
        P2P_TRY_CUDA(cudaMemset2DAsync(out, (size_t)ld * 8, 0, (size_t)nrhs * 8, (size_t)plan->n, s), "p2p_apply/zero");
    if (plan->n_items == 0) return P2P_OK;
    if (is_multi(plan, nrhs, path)) return p2p_multi_launch(plan, (float2*)out, nrhs, ld, a.k, s);
    const int R = path == P2P_PATH_FP32_PER_RHS ? 1 : (nrhs >= 4 ? 4 : (nrhs >= 2 ? 2 : 1));
    return R == 1 ? launch_pair<1>(plan, a, s) : (R == 2 ? launch_pair<2>(plan, a, s) : launch_pair<4>(plan, a, s));
}

P2P_API p2p_status p2p_apply_path(const p2p_plan* plan, const void* lambda, void* out, int32_t nrhs, int64_t ld,
                                  int32_t adjoint, p2p_path path, p2p_stream_t stream) {
    p2p_status st = check_apply_args(plan, lambda, out, nrhs, ld);
    if (st != P2P_OK) return st;
    if (lambda == out && plan->n > 0 && plan->n_src > 0) return P2P_ERR_INVALID;
    st = p2p_apply_stage(plan, lambda, nrhs, ld, path, stream);
    if (st != P2P_OK) return st;
    return p2p_apply_staged(plan, out, nrhs, ld, adjoint, path, stream);
}

P2P_API p2p_status p2p_apply(const p2p_plan* plan, const void* lambda, void* out, int32_t nrhs, int64_t ld,
                             p2p_stream_t stream) {
    return p2p_apply_path(plan, lambda, out, nrhs, ld, 0, P2P_PATH_AUTO, stream);
}

P2P_API p2p_status p2p_apply_adjoint(const p2p_plan* plan, const void* g, void* out, int32_t nrhs, int64_t ld,
                                     p2p_stream_t stream) {
    // a two-set operator's adjoint maps target space to source space: a plan with the roles exchanged
    if (plan && plan->two_sets) return P2P_ERR_UNSUPPORTED;
    return p2p_apply_path(plan, g, out, nrhs, ld, 1, P2P_PATH_AUTO, stream);
}

P2P_API p2p_status p2p_grad_points(const p2p_plan* plan, const void* lambda, const void* g, float* grad,
                                   int32_t nrhs, int64_t ld, p2p_stream_t stream) {
    p2p_status st = check_apply_args(plan, lambda, g, nrhs, ld);
    if (st != P2P_OK) return st;
    if (plan->n == 0) return P2P_OK;
    if (!grad || ((uintptr_t)grad & 3)) return P2P_ERR_INVALID;
    if (plan->layout == P2P_LAYOUT_SYMMETRIC) return P2P_ERR_UNSUPPORTED;  // needs the full source lists
    if (plan->two_sets) return P2P_ERR_UNSUPPORTED;                         // one point set only
    return p2p_grad_launch(plan, (const float2*)lambda, (const float2*)g, grad, nrhs, ld, (cudaStream_t)stream);
}

}  // extern "C"
