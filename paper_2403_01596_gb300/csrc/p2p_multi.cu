// Several right-hand sides in FP32: the near-field sum of 2 .. 8 right-hand sides
// per launch with G evaluated once for all of them.
//
// What bounds it.  A pair costs 3 MUFU operations and ~14 FP32 ones for G, and 4
// FP32 operations per right-hand side, so from four right-hand sides on the FMA
// pipe is the limit (46 lane operations per pair at eight: 0.16 ms for the
// 1.4e8 pairs of a 500 000-point assembly on 152 SMs).  The staged pipeline
// (p2p_pair.cuh) spends more than that around it: at four right-hand sides its two
// stages of a whole 192-source chunk take 25 KB per warp, so 8 warps fill an SM, eight
// right-hand sides are two sweeps that form G twice, and their strengths are
// loaded synchronously.
//
// Here an item (target box, source chunk) streams through the warp in sub-chunks
// of at most 64 sources, three steps deep -- source indices in registers,
// coordinates and strengths in flight into one half of the warp's buffer
// (cp.async), the sweep on the other half -- and the accumulators stay in registers
// across the sub-chunks: 5 KB of shared memory per warp at two right-hand sides, 12 KB at
// eight, 16 or 12 warps per SM.  The stream runs on over target groups and items, so the next item's
// first sources are on their way while this one's slices are summed.
//
// Strengths are staged by blocks of right-hand sides, a row per source with the real
// parts before the imaginary parts, so that the complex multiply-add runs on the
// packed two-lane FP32 instructions over pairs of right-hand sides without moves; the
// distances run packed over pairs of targets.  Every packed operation rounds as its
// scalar counterpart in pair_core, in the same order.
//
// Measured on one GB300, applies including the staging, against the staged pipeline at 4 right-hand sides per sweep:
// the 500 000-point assembly with 8 right-hand sides 0.41 ms (0.90), 300 001 points on a sphere at 47 per box with 5
// 0.44 ms (0.79), with 12 (Laplace) 0.51 ms (0.87), at 7 per box with 3 in the redundant layout 0.10 ms (0.32: no
// per-box repack of the strengths), 10 371 points with 2 23 us (30).
#include <algorithm>

#include "p2p_pair.cuh"

using namespace p2p_detail;
using namespace p2p_pair;

namespace {

// Sources of a sub-chunk at most.  A sub-chunk costs ~150 instructions around its sweep, which weigh most where a pair
// costs little: 64 instead of 32 took 3 right-hand sides on 200 001 points from 75 to 71 us and the Laplace gradient on
// 500 001 points from 120 to 107 us, and changed 8 right-hand sides by 1 % at most.
constexpr int kSub = 64;
constexpr int kLaneSrc = kSub / 32;     // of which a lane copies
constexpr int kBlockRhs = 8;            // right-hand sides per launch at most

// Warps of an SM: two blocks of 8 at 128 registers, or one of 12 at 168 where that is faster although fewer warps are
// resident: 8 right-hand sides (which spill at 128) 424 -> 417 us on the 500 000-point assembly and 225 -> 218 us on
// 300 001 sphere points, the Helmholtz gradient 550 -> 516 us on 500 001 points at 50 per box; the Laplace gradient
// (107 -> 116 us on 500 001 points at 8), the Helmholtz gradient of uneven geometries (p2p_grad_launch) and 3 right-hand
// sides (71 -> 80 us) are slower with 12.
struct Shape {
    int warps, blocks;
};
__host__ __device__ constexpr Shape multi_shape(int R) { return R == 8 ? Shape{12, 1} : Shape{8, 2}; }

struct MultiArgs {
    const ItemRec* items;
    int32_t n_items;
    const float4* xs;       // box-sorted source coordinates
    const float4* xt;       // box-sorted target coordinates
    const int32_t* nb_src;  // per-box source lists (box-sorted indices)
    const float* lam;       // staged strengths of this block: 2R floats per source
    const int32_t* perm;
    float2* out;            // first right-hand side of this block
    int64_t ld;
    int32_t nrhs;           // right-hand sides of this block (<= R)
    float k;
    int32_t tg;
    int32_t atomic_out;
};

__host__ __device__ constexpr int stage_floats(int R) { return kSub * (4 + 2 * R); }
__host__ __device__ constexpr int warp_floats(int R) { return 2 * stage_floats(R) + 32 * 2 * R; }

// A place in the warp's stream of sub-chunks: the item, its target group and the group's sub-chunk.
struct Place {
    int32_t src_off, ns, tb, nt, m_end, map_full, map_last;  // of the item (ItemRec)
    int32_t item;   // index in the item list (>= n_items: the stream has ended)
    int t0, s0;
    int32_t map;
    int len;        // sources of the sub-chunk: whole rounds of the map's Q slices
};

__device__ __forceinline__ void set_item(Place& p, int32_t rec) {
    p.src_off = __shfl_sync(P2P_FULL_MASK, rec, 0);
    p.ns = __shfl_sync(P2P_FULL_MASK, rec, 1);
    p.tb = __shfl_sync(P2P_FULL_MASK, rec, 2);
    p.nt = __shfl_sync(P2P_FULL_MASK, rec, 3);
    p.m_end = __shfl_sync(P2P_FULL_MASK, rec, 4) & 0xFFFF;
    p.map_full = __shfl_sync(P2P_FULL_MASK, rec, 5);
    p.map_last = __shfl_sync(P2P_FULL_MASK, rec, 6);
}
__device__ __forceinline__ void set_group(Place& p, int tg) {
    p.map = p.t0 + tg >= p.nt ? p.map_last : p.map_full;
}
__device__ __forceinline__ void set_len(Place& p) {
    const int Q = map_q(p.map);
    p.len = min(p.ns - p.s0, (kSub / Q) * Q);
}

// Sorted source indices of a sub-chunk, a lane's own.
struct Sources {
    int32_t v[kLaneSrc];
};

template <int R>
struct Stream {
    const MultiArgs& a;
    int lane;
    int32_t worker, workers, turn;
    int32_t rec;      // record of the item after the latest place's, field f in lane f
    int32_t rec_item;
    float* base;

    __device__ __forceinline__ float* buf(int h) const { return base + h * stage_floats(R); }
    __device__ __forceinline__ Place first(int32_t item) {
        Place p;
        p.item = item;
        set_item(p, load_rec_lane(a.items, item, a.n_items, lane));
        rec_item = (int32_t)min((int64_t)a.n_items, p2p_turn(++turn, worker, workers));
        rec = load_rec_lane(a.items, rec_item, a.n_items, lane);
        p.t0 = p.s0 = 0;
        set_group(p, a.tg);
        set_len(p);
        return p;
    }
    __device__ __forceinline__ Place next(const Place& c) {
        Place p = c;
        p.s0 += p.len;
        if (p.s0 >= p.ns) {
            p.s0 = 0;
            p.t0 += a.tg;
            if (p.t0 >= p.nt) {
                p.t0 = 0;
                p.item = rec_item;
                if (p.item < a.n_items) {
                    set_item(p, rec);
                    rec_item = (int32_t)min((int64_t)a.n_items, p2p_turn(++turn, worker, workers));
                    rec = load_rec_lane(a.items, rec_item, a.n_items, lane);
                }
            }
            set_group(p, a.tg);
        }
        set_len(p);
        return p;
    }
    __device__ __forceinline__ Sources index(const Place& p) const {
        Sources j;
#pragma unroll
        for (int i = 0; i < kLaneSrc; ++i)
            j.v[i] = p.item < a.n_items && 32 * i + lane < p.len ? __ldg(a.nb_src + p.src_off + p.s0 + 32 * i + lane) : 0;
        return j;
    }
    // copies of the sub-chunk at p (lane's sources j) into half h; one group per call, possibly empty
    __device__ __forceinline__ void copy(const Place& p, const Sources& j, int h) const {
#pragma unroll
        for (int c = 0; c < kLaneSrc; ++c) {
            const int l = 32 * c + lane;
            if (p.item < a.n_items && l < p.len) {
                cp_async16(buf(h) + 4 * l, a.xs + j.v[c]);
                float* dst = buf(h) + 4 * kSub + 2 * R * l;
                const float* src = a.lam + (int64_t)j.v[c] * (2 * R);
#pragma unroll
                for (int i = 0; i < 2 * R; i += 4) cp_async16(dst + i, src + i);
            }
        }
        cp_async_commit();
    }
};

// One source against the lane's TT targets (negated coordinates), R right-hand sides.  own: a source of the targets'
// own cell, where r = 0 gives nothing; other sources start r^2 at the smallest normal float (pair_core).
template <int KERN, int R, int TT>
__device__ __forceinline__ void multi_core(const float4 p, const float* __restrict__ l, bool own, const float (&nx)[TT],
                                           const float (&ny)[TT], const float (&nz)[TT], float2 (&re)[TT][R / 2],
                                           float2 (&im)[TT][R / 2], float k) {
    float2 lr[R / 2], li[R / 2];
    if constexpr (R == 2) {
        const float4 v = *reinterpret_cast<const float4*>(l);
        lr[0] = make_float2(v.x, v.y);
        li[0] = make_float2(v.z, v.w);
    } else {
#pragma unroll
        for (int i = 0; i < R / 4; ++i) {
            const float4 v = reinterpret_cast<const float4*>(l)[i], w = reinterpret_cast<const float4*>(l + R)[i];
            lr[2 * i] = make_float2(v.x, v.y);
            lr[2 * i + 1] = make_float2(v.z, v.w);
            li[2 * i] = make_float2(w.x, w.y);
            li[2 * i + 1] = make_float2(w.z, w.w);
        }
    }
    const float base = own ? 0.f : 1.17549435e-38f;
    float gr[TT], gi[TT];
    if constexpr (TT % 2 == 0) {
        const float2 px = make_float2(p.x, p.x), py = make_float2(p.y, p.y), pz = make_float2(p.z, p.z);
#pragma unroll
        for (int u = 0; u < TT; u += 2) {
            const float2 dx = __fadd2_rn(px, make_float2(nx[u], nx[u + 1]));
            const float2 dy = __fadd2_rn(py, make_float2(ny[u], ny[u + 1]));
            const float2 dz = __fadd2_rn(pz, make_float2(nz[u], nz[u + 1]));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, make_float2(base, base))));
            float2 inv = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            inv.x = r2.x > 0.f ? inv.x : 0.f;
            inv.y = r2.y > 0.f ? inv.y : 0.f;
            if (KERN == P2P_HELMHOLTZ) {
                const float2 ph = __fmul2_rn(make_float2(k, k), __fmul2_rn(r2, inv));
                float2 sn, cs;
                __sincosf(ph.x, &sn.x, &cs.x);
                __sincosf(ph.y, &sn.y, &cs.y);
                const float2 r = __fmul2_rn(cs, inv), i = __fmul2_rn(sn, inv);
                gr[u] = r.x;
                gr[u + 1] = r.y;
                gi[u] = i.x;
                gi[u + 1] = i.y;
            } else {
                gr[u] = inv.x;
                gr[u + 1] = inv.y;
            }
        }
    } else {
        const float dx = p.x + nx[0], dy = p.y + ny[0], dz = p.z + nz[0];
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, base)));
        float inv = rsqrtf(r2);
        inv = r2 > 0.f ? inv : 0.f;
        if (KERN == P2P_HELMHOLTZ) {
            float sn, cs;
            __sincosf(k * (r2 * inv), &sn, &cs);
            gr[0] = cs * inv;
            gi[0] = sn * inv;
        } else {
            gr[0] = inv;
        }
    }
#pragma unroll
    for (int u = 0; u < TT; ++u) {
        const float2 g = make_float2(gr[u], gr[u]);
        if (KERN == P2P_HELMHOLTZ) {
            const float2 h = make_float2(gi[u], gi[u]), nh = make_float2(-gi[u], -gi[u]);
#pragma unroll
            for (int i = 0; i < R / 2; ++i) {
                re[u][i] = __ffma2_rn(g, lr[i], __ffma2_rn(nh, li[i], re[u][i]));
                im[u][i] = __ffma2_rn(g, li[i], __ffma2_rn(h, lr[i], im[u][i]));
            }
        } else {
#pragma unroll
            for (int i = 0; i < R / 2; ++i) {
                re[u][i] = __ffma2_rn(g, lr[i], re[u][i]);
                im[u][i] = __ffma2_rn(g, li[i], im[u][i]);
            }
        }
    }
}

// The target group at `cur` (whose sub-chunk is on its way into half h) through all of its sub-chunks: pair(p, l, own)
// for the sources of the lane's slice q of Q, own: a source of the targets' own cell.  nxt: the place after cur, its
// indices in j.  Leaves cur, nxt, j and h at the next group's first sub-chunk.
template <int R, typename Pair>
__device__ __forceinline__ void sweep_stream(Stream<R>& st, Place& cur, Place& nxt, Sources& j, int& h, int q, int Q, Pair pair) {
    const int m_end = cur.m_end;
    while (true) {
        st.copy(nxt, j, h ^ 1);
        const Place after = nxt.item < st.a.n_items ? st.next(nxt) : nxt;
        const Sources ja = st.index(after);
        cp_async_wait<1>();
        __syncwarp();
        if (q < Q) {
            const float* buf = st.buf(h);
            const int own = m_end - cur.s0;
            for (int s = q; s < cur.len; s += Q)
                pair(*reinterpret_cast<const float4*>(buf + 4 * s), buf + 4 * kSub + 2 * R * s, s < own);
        }
        __syncwarp();  // the half is read before the copies of the place after next overwrite it
        const bool last = cur.s0 + cur.len >= cur.ns;
        cur = nxt;
        nxt = after;
        j = ja;
        h ^= 1;
        if (last) break;
    }
}

// One target group (sweep_stream) and its results.
template <int KERN, int R, int TT>
__device__ __forceinline__ void run_group(Stream<R>& st, Place& cur, Place& nxt, Sources& j, int& h, float* red) {
    const MultiArgs& a = st.a;
    const int lane = st.lane;
    const int32_t map = cur.map;
    const int G = map_g(map), Q = map_q(map), q = map_div(map, lane), g = lane - q * G;
    const int tb = cur.tb + cur.t0, nt = min(a.tg, cur.nt - cur.t0);
    const int32_t perm0 = lane < nt ? __ldg(a.perm + tb + lane) : 0;
    float nx[TT], ny[TT], nz[TT];
    float2 re[TT][R / 2], im[TT][R / 2];
#pragma unroll
    for (int u = 0; u < TT; ++u) {
        const int t = g + u * G;
        const float4 x = t < nt && q < Q ? __ldg(a.xt + tb + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        nx[u] = -x.x;
        ny[u] = -x.y;
        nz[u] = -x.z;
#pragma unroll
        for (int i = 0; i < R / 2; ++i) re[u][i] = im[u][i] = make_float2(0.f, 0.f);
    }
    sweep_stream<R>(st, cur, nxt, j, h, q, Q, [&](const float4& p, const float* l, bool own) {
        multi_core<KERN, R, TT>(p, l, own, nx, ny, nz, re, im, a.k);
    });
    // slice partials -> results, one target of every lane at a time: (Re, Re, Im, Im) of two right-hand sides per
    // 16 bytes, lane after lane
    float4* red4 = reinterpret_cast<float4*>(red);
#pragma unroll
    for (int u = 0; u < TT; ++u) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) red4[i * 32 + lane] = make_float4(re[u][i].x, re[u][i].y, im[u][i].x, im[u][i].y);
        __syncwarp();
        const int here = min(G, nt - u * G);  // targets u G .. u G + here - 1
        for (int e0 = 0; e0 < G * (R / 2); e0 += 32) {
            const int e = e0 + lane;
            const int i = min(map_div(map, min(e, 127)), R / 2 - 1), gg = e - i * G;
            const bool on = e < G * (R / 2) && gg < here;
            const int t = u * G + gg;
            int32_t row = __shfl_sync(P2P_FULL_MASK, perm0, t & 31);
            if (!on) continue;
            if (t >= 32) row = __ldg(a.perm + tb + t);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int qq = 0; qq < Q; ++qq) {
                const float4 w = red4[i * 32 + qq * G + gg];
                v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
            }
            float2* dst = a.out + (int64_t)row * a.ld + 2 * i;
            const float2 o0 = make_float2(v.x * kInv4Pi, v.z * kInv4Pi), o1 = make_float2(v.y * kInv4Pi, v.w * kInv4Pi);
            if (2 * i < a.nrhs) {
                if (a.atomic_out) atomicAdd(dst, o0);
                else dst[0] = o0;
            }
            if (2 * i + 1 < a.nrhs) {
                if (a.atomic_out) atomicAdd(dst + 1, o1);
                else dst[1] = o1;
            }
        }
        __syncwarp();
    }
}

template <int KERN, int R>
__global__ void __launch_bounds__(multi_shape(R).warps * 32, multi_shape(R).blocks)
    k_pair_multi(const __grid_constant__ MultiArgs a) {
    constexpr int kWarps = multi_shape(R).warps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* ws = reinterpret_cast<float*>(smem_raw) + warp * warp_floats(R);
    Stream<R> st{a, lane, (int32_t)(blockIdx.x * kWarps + warp), (int32_t)gridDim.x * kWarps, 0, 0, 0, ws};
    float* red = ws + 2 * stage_floats(R);
    const int32_t item = (int32_t)blockIdx.x * kWarps + warp;
    if (item >= a.n_items) return;
    Place cur = st.first(item);
    st.copy(cur, st.index(cur), 0);
    Place nxt = st.next(cur);
    Sources j = st.index(nxt);
    int h = 0;
    while (cur.item < a.n_items) {
        const int tt = map_tt(cur.map);
        if (tt == 1) run_group<KERN, R, 1>(st, cur, nxt, j, h, red);
        else if (tt == 2) run_group<KERN, R, 2>(st, cur, nxt, j, h, red);
        else run_group<KERN, R, 4>(st, cur, nxt, j, h, red);
    }
    cp_async_wait<0>();
}

// ------------------------------------------------------ coordinate gradient --

// The derivative with respect to the target's coordinates, one right-hand side per launch.  A pair is 3 MUFU and ~30
// FP32 operations (19 of them on the packed instructions), so both pipes and the issue slots are about equally busy;
// what the kernel must avoid is standing still.  One item per warp, staged whole and synchronously before its sweep,
// left 18 warps per SM waiting for two dependent gathers at every item.  Here the rows (lambda, g) come through the
// same stream as the strengths of two right-hand sides (at 80 registers, 24 warps, the sweep spills and takes 13 %
// longer than with 16 warps); one launch stages both inputs and zeroes the result.  Staging included: 262 144 points on
// a sphere at 16 per box 147 -> 118 us, Laplace on 500 001 points of an ellipsoid at 8 160 -> 107 us, 12 001 points at
// 10 31 -> 22 us, 500 001 points at 50 554 -> 516 us.
constexpr int kGradWarpFloats = 2 * stage_floats(2) + 32 * kMaxTT * 4;

// One source against the lane's TT targets (negated coordinates; strengths and upstream values tl, tg).
template <int KERN, int TT>
__device__ __forceinline__ void grad_core(const float4 p, const float4 lg, const float (&nx)[TT], const float (&ny)[TT],
                                          const float (&nz)[TT], const float2 (&tl)[TT], const float2 (&tg)[TT],
                                          float (&acc)[TT][3], float k) {
    // with d = source - target: grad = w d, w = (G'(r) / r) C, C = conj(g_t) lambda_s + conj(g_s) lambda_t
    if constexpr (TT % 2 == 0) {
        const float2 px = make_float2(p.x, p.x), py = make_float2(p.y, p.y), pz = make_float2(p.z, p.z);
        const float2 lx = make_float2(lg.x, lg.x), ly = make_float2(lg.y, lg.y), gx = make_float2(lg.z, lg.z),
                     gy = make_float2(lg.w, lg.w);
        const float2 nlx = make_float2(-lg.x, -lg.x), ngy = make_float2(-lg.w, -lg.w);
#pragma unroll
        for (int u = 0; u < TT; u += 2) {
            const float2 dx = __fadd2_rn(px, make_float2(nx[u], nx[u + 1]));
            const float2 dy = __fadd2_rn(py, make_float2(ny[u], ny[u + 1]));
            const float2 dz = __fadd2_rn(pz, make_float2(nz[u], nz[u + 1]));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            float2 inv = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            inv.x = r2.x > 0.f ? inv.x : 0.f;
            inv.y = r2.y > 0.f ? inv.y : 0.f;
            const float2 inv2 = __fmul2_rn(inv, inv);
            const float2 tlx = make_float2(tl[u].x, tl[u + 1].x), tly = make_float2(tl[u].y, tl[u + 1].y);
            const float2 tgx = make_float2(tg[u].x, tg[u + 1].x), tgy = make_float2(tg[u].y, tg[u + 1].y);
            const float2 cr = __ffma2_rn(tgx, lx, __ffma2_rn(tgy, ly, __ffma2_rn(gx, tlx, __fmul2_rn(gy, tly))));
            float2 w;
            if (KERN == P2P_HELMHOLTZ) {
                const float2 ci = __ffma2_rn(tgx, ly, __ffma2_rn(tgy, nlx, __ffma2_rn(gx, tly, __fmul2_rn(ngy, tlx))));
                const float2 kr = __fmul2_rn(make_float2(k, k), __fmul2_rn(r2, inv));
                float2 sn, cs;
                __sincosf(kr.x, &sn.x, &cs.x);
                __sincosf(kr.y, &sn.y, &cs.y);
                // -G' r^2 = (cos + kr sin) + i (sin - kr cos), the sign goes into d
                const float2 a = __ffma2_rn(sn, kr, cs);
                const float2 b = __ffma2_rn(make_float2(-cs.x, -cs.y), kr, sn);
                w = __ffma2_rn(a, cr, __fmul2_rn(make_float2(-b.x, -b.y), ci));
                w = __fmul2_rn(w, inv2);
            } else {
                w = __fmul2_rn(inv2, cr);
            }
            w = __fmul2_rn(w, inv);
            float2 ax = make_float2(acc[u][0], acc[u + 1][0]), ay = make_float2(acc[u][1], acc[u + 1][1]),
                   az = make_float2(acc[u][2], acc[u + 1][2]);
            ax = __ffma2_rn(w, dx, ax);
            ay = __ffma2_rn(w, dy, ay);
            az = __ffma2_rn(w, dz, az);
            acc[u][0] = ax.x;
            acc[u + 1][0] = ax.y;
            acc[u][1] = ay.x;
            acc[u + 1][1] = ay.y;
            acc[u][2] = az.x;
            acc[u + 1][2] = az.y;
        }
    } else {
        const float dx = p.x + nx[0], dy = p.y + ny[0], dz = p.z + nz[0];
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        float inv = rsqrtf(r2);
        inv = r2 > 0.f ? inv : 0.f;
        const float cr = fmaf(tg[0].x, lg.x, fmaf(tg[0].y, lg.y, fmaf(lg.z, tl[0].x, lg.w * tl[0].y)));
        float w = cr;
        if (KERN == P2P_HELMHOLTZ) {
            const float ci = fmaf(tg[0].x, lg.y, fmaf(tg[0].y, -lg.x, fmaf(lg.z, tl[0].y, -lg.w * tl[0].x)));
            const float kr = k * (r2 * inv);
            float sn, cs;
            __sincosf(kr, &sn, &cs);
            w = fmaf(fmaf(sn, kr, cs), cr, -fmaf(-cs, kr, sn) * ci);
        }
        w = w * (inv * inv) * inv;
        acc[0][0] = fmaf(w, dx, acc[0][0]);
        acc[0][1] = fmaf(w, dy, acc[0][1]);
        acc[0][2] = fmaf(w, dz, acc[0][2]);
    }
}

// One target group of the gradient: its sums are added to the (zeroed) result.
template <int KERN, int TT>
__device__ __forceinline__ void run_grad(Stream<2>& st, Place& cur, Place& nxt, Sources& j, int& h, float* red, float* out) {
    const MultiArgs& a = st.a;
    const int lane = st.lane;
    const int32_t map = cur.map;
    const int G = map_g(map), Q = map_q(map), q = map_div(map, lane), g = lane - q * G;
    const int tb = cur.tb + cur.t0, nt = min(a.tg, cur.nt - cur.t0);
    const int32_t perm0 = lane < nt ? __ldg(a.perm + tb + lane) : 0;
    float nx[TT], ny[TT], nz[TT], acc[TT][3];
    float2 tl[TT], tg[TT];
#pragma unroll
    for (int u = 0; u < TT; ++u) {
        const int t = g + u * G;
        const bool on = t < nt && q < Q;
        const float4 x = on ? __ldg(a.xt + tb + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 v = on ? __ldg(reinterpret_cast<const float4*>(a.lam) + tb + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        nx[u] = -x.x;
        ny[u] = -x.y;
        nz[u] = -x.z;
        tl[u] = make_float2(v.x, v.y);
        tg[u] = make_float2(v.z, v.w);
        acc[u][0] = acc[u][1] = acc[u][2] = 0.f;
    }
    sweep_stream<2>(st, cur, nxt, j, h, q, Q, [&](const float4& p, const float* l, bool) {
        grad_core<KERN, TT>(p, *reinterpret_cast<const float4*>(l), nx, ny, nz, tl, tg, acc, a.k);
    });
    float4* red4 = reinterpret_cast<float4*>(red);
#pragma unroll
    for (int u = 0; u < TT; ++u) red4[u * 32 + lane] = make_float4(acc[u][0], acc[u][1], acc[u][2], 0.f);
    __syncwarp();
    for (int t = lane; t < nt; t += 32) {
        const int u = map_div(map, t), gg = t - u * G;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int qq = 0; qq < Q; ++qq) {
            const float4 w = red4[u * 32 + qq * G + gg];
            v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, 0.f);
        }
        float* dst = out + (int64_t)(t == lane ? perm0 : __ldg(a.perm + tb + t)) * 3;
        atomicAdd(dst, v.x * kInv4Pi);
        atomicAdd(dst + 1, v.y * kInv4Pi);
        atomicAdd(dst + 2, v.z * kInv4Pi);
    }
    __syncwarp();
}

// WARPS: of a block, 12 (one block per SM) or 8 (two).
template <int KERN, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS == 12 ? 1 : 2) k_grad(const __grid_constant__ MultiArgs a, float* out) {
    constexpr int kWarps = WARPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* ws = reinterpret_cast<float*>(smem_raw) + warp * kGradWarpFloats;
    Stream<2> st{a, lane, (int32_t)(blockIdx.x * kWarps + warp), (int32_t)gridDim.x * kWarps, 0, 0, 0, ws};
    float* red = ws + 2 * stage_floats(2);
    const int32_t item = (int32_t)blockIdx.x * kWarps + warp;
    if (item >= a.n_items) return;
    Place cur = st.first(item);
    st.copy(cur, st.index(cur), 0);
    Place nxt = st.next(cur);
    Sources j = st.index(nxt);
    int h = 0;
    while (cur.item < a.n_items) {
        const int tt = map_tt(cur.map);
        if (tt == 1) run_grad<KERN, 1>(st, cur, nxt, j, h, red, out);
        else if (tt == 2) run_grad<KERN, 2>(st, cur, nxt, j, h, red, out);
        else run_grad<KERN, 4>(st, cur, nxt, j, h, red, out);
    }
    cp_async_wait<0>();
}

// dst[q * n + s] = (lambda, g)[rows[s] * ld + q], and the result's 3 n floats zeroed.
__global__ void k_grad_stage(const float2* __restrict__ lam, const float2* __restrict__ g, int64_t ld,
                             const int32_t* __restrict__ rows, int64_t n, int32_t nrhs, float4* __restrict__ dst,
                             float* __restrict__ grad) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int64_t row = (int64_t)rows[s] * ld;
    for (int q = 0; q < nrhs; ++q) {
        const float2 a = lam[row + q], b = g[row + q];
        dst[q * n + s] = make_float4(a.x, a.y, b.x, b.y);
    }
    if (grad)
        for (int i = 0; i < 3; ++i) grad[i * n + s] = 0.f;
}

// Right-hand sides of a launch (2, 4 or 8 accumulators) for the `left` ones still to do.
__host__ __device__ inline int block_width(int left) { return left > 4 ? 8 : (left > 2 ? 4 : 2); }

// All blocks of the right-hand sides, one after the other (kBlockRhs wide, the last one as wide as its launch): 2R floats
// per source, Re of the block's right-hand sides, then Im (zero past nrhs).  One thread per source and column.
__global__ void k_multi_stage(const float2* __restrict__ src, int64_t ld, const int32_t* __restrict__ rows, int64_t n,
                              int32_t nrhs, int32_t columns, float* __restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * columns) return;
    const int64_t s = i / columns;
    const int c = (int)(i - s * columns), b = c & ~(kBlockRhs - 1), r = c - b;
    const int R = block_width(min(kBlockRhs, nrhs - b));
    const float2 v = c < nrhs ? src[(int64_t)rows[s] * ld + c] : make_float2(0.f, 0.f);
    float* d = dst + n * 2 * b + s * 2 * R + r;
    d[0] = v.x;
    d[R] = v.y;
}

using MultiKernel = void (*)(MultiArgs);
MultiKernel multi_kernel(const p2p_plan* p, int R) {
    if (p->kernel == P2P_HELMHOLTZ)
        return R == 8 ? k_pair_multi<P2P_HELMHOLTZ, 8> : (R == 4 ? k_pair_multi<P2P_HELMHOLTZ, 4> : k_pair_multi<P2P_HELMHOLTZ, 2>);
    return R == 8 ? k_pair_multi<P2P_LAPLACE, 8> : (R == 4 ? k_pair_multi<P2P_LAPLACE, 4> : k_pair_multi<P2P_LAPLACE, 2>);
}

}  // namespace

// Staged columns (complex) of nrhs right-hand sides: every block rounded up to its width.
int32_t p2p_multi_columns(int32_t nrhs) {
    if (nrhs <= 1) return nrhs;
    int c = 0;
    for (int b = 0; b < nrhs; b += kBlockRhs) c += block_width(std::min(kBlockRhs, nrhs - b));
    return c;
}

// Persistent grids for 2, 4 and 8 right-hand sides per launch.
cudaError_t p2p_multi_configure(p2p_plan* p) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int i = 0; i < 3 && e == cudaSuccess; ++i) {
        const int R = 2 << i, warps = multi_shape(R).warps, smem = warps * warp_floats(R) * (int)sizeof(float);
        int per_sm = 0;
        MultiKernel kern = multi_kernel(p, R);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem);
        p->multi_grid[i] = e == cudaSuccess ? per_sm * sms : 0;
    }
    return e;
}

p2p_status p2p_multi_stage(const p2p_plan* p, const float2* lam, int32_t nrhs, int64_t ld, cudaStream_t s) {
    const int32_t columns = p2p_multi_columns(nrhs);
    k_multi_stage<<<(unsigned)((p->n_src * columns + 255) / 256), 256, 0, s>>>(lam, ld, p->src_perm, p->n_src, nrhs, columns,
                                                                              reinterpret_cast<float*>(p->lam_buf));
    P2P_CHECK_LAUNCH("p2p_apply_stage/multi");
    return P2P_OK;
}

// Results are stored where a box's list is one chunk, else added (the caller has zeroed them).
p2p_status p2p_multi_launch(const p2p_plan* p, float2* out, int32_t nrhs, int64_t ld, float k, cudaStream_t s) {
    MultiArgs a;
    a.items = p->items;
    a.n_items = (int32_t)p->n_items;
    a.xs = p->xs_src;
    a.xt = p->xs;
    a.nb_src = p->nb_src;
    a.lam = reinterpret_cast<const float*>(p->lam_buf);
    a.perm = p->perm;
    a.ld = ld;
    a.k = k;
    a.tg = p->tune.target_group;
    a.atomic_out = p->max_chunks > 1;
    for (int b = 0; b < nrhs; b += kBlockRhs) {
        a.nrhs = std::min(kBlockRhs, nrhs - b);
        const int R = block_width(a.nrhs), warps = multi_shape(R).warps, smem = warps * warp_floats(R) * (int)sizeof(float);
        const int grid = (int)std::min<int64_t>(p->multi_grid[R == 8 ? 2 : R / 4], ((int64_t)a.n_items + warps - 1) / warps);
        if (grid <= 0) return P2P_ERR_UNSUPPORTED;
        a.out = out + b;
        multi_kernel(p, R)<<<grid, warps * 32, smem, s>>>(a);
        P2P_CHECK_LAUNCH("p2p_apply/multi");
        a.lam += p->n_src * 2 * R;
    }
    return P2P_OK;
}

// The coordinate gradient (one point set), added up over the right-hand sides.
p2p_status p2p_grad_launch(const p2p_plan* p, const float2* lam, const float2* g, float* grad, int32_t nrhs, int64_t ld,
                           cudaStream_t s) {
    int dev = 0, sms = 0;
    P2P_TRY_CUDA(cudaGetDevice(&dev), "p2p_grad_points/device");
    P2P_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "p2p_grad_points/device");
    float4* rows = reinterpret_cast<float4*>(p->lam_buf);
    // a result that overlaps an input is zeroed once all of it has been staged
    const char *lo = reinterpret_cast<const char*>(grad), *hi = lo + (size_t)p->n * 3 * sizeof(float);
    const size_t in_bytes = ((size_t)(p->n - 1) * ld + nrhs) * sizeof(float2);
    bool overlap = false;
    for (const char* v : {reinterpret_cast<const char*>(lam), reinterpret_cast<const char*>(g)})
        overlap |= v < hi && lo < v + in_bytes;
    k_grad_stage<<<(unsigned)((p->n + 255) / 256), 256, 0, s>>>(lam, g, ld, p->perm, p->n, nrhs, rows,
                                                               overlap ? nullptr : grad);
    P2P_CHECK_LAUNCH("p2p_grad_points/stage");
    if (overlap) P2P_TRY_CUDA(cudaMemsetAsync(grad, 0, (size_t)p->n * 3 * sizeof(float), s), "p2p_grad_points/zero");
    MultiArgs a{};
    a.items = p->items;
    a.n_items = (int32_t)p->n_items;
    a.xs = p->xs_src;
    a.xt = p->xs;
    a.nb_src = p->nb_src;
    a.perm = p->perm;
    a.k = p->k;
    a.tg = p->tune.target_group;
    // Where the heaviest box is worth more than four of the average warps (32 per SM), the items' turns leave the warps with
    // its items far behind the others: a grid of sixteen times the resident blocks, whose blocks come as SMs become free.
    // Helmholtz takes 16 warps per SM there, more of them beside the long ones.  Clustered assemblies, as before the stream /
    // with 12 warps in turns / here, us: 60 001 points at 10 per box 75 / 73 / 64, at 60 161 / 189 / 148, 300 001 at 10 230 / 249 /
    // 212, Laplace 150 / 149 / 130.  On even geometries the larger grid only starts more blocks (262 144 sphere points at 16,
    // Helmholtz with 12 warps 119 -> 127; a cube at 20 176 -> 196).
    const bool uneven = p->heavy > 4 * p->even;
    const bool helm = p->kernel == P2P_HELMHOLTZ, narrow = helm && !uneven;
    const Shape shape = narrow ? Shape{12, 1} : Shape{8, 2};
    const int64_t blocks = ((int64_t)a.n_items + shape.warps - 1) / shape.warps;
    if (blocks == 0) return P2P_OK;
    const int smem = shape.warps * kGradWarpFloats * (int)sizeof(float);
    auto kern = narrow ? k_grad<P2P_HELMHOLTZ, 12> : (helm ? k_grad<P2P_HELMHOLTZ, 8> : k_grad<P2P_LAPLACE, 8>);
    const int64_t grid = std::min<int64_t>(blocks, (int64_t)sms * shape.blocks * (uneven ? 16 : 1));
    if (smem > 48 * 1024)
        P2P_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "p2p_grad_points");
    for (int q = 0; q < nrhs; ++q) {
        a.lam = reinterpret_cast<const float*>(rows + (int64_t)q * p->n);
        kern<<<(unsigned)grid, shape.warps * 32, smem, s>>>(a, grad);
        P2P_CHECK_LAUNCH("p2p_grad_points/kernel");
    }
    return P2P_OK;
}
