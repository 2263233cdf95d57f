// Multi-RHS P2P on the 5th-generation tensor cores (tcgen05, TMEM operands).
//
// Contraction.  A unit of work is a window of up to 128 box-sorted targets (the
// rows of one MMA), an entry one group of 16 consecutive box-sorted sources.  For
// every entry with a source near one of the unit's targets two real MMA chains add
//
//     D1[128 x 2R] += Gr[128 x 16] . [Lr | Li][16 x 2R]
//     D2[128 x 2R] += Gi[128 x 16] . [Lr | Li][16 x 2R]
//
// with Gr, Gi = Re, Im G(x_t, y_s) (0 where s is not in t's neighbourhood or r = 0)
// and Lr, Li = Re, Im lambda[s, r], so that Re out[t, r] = D1[t, r] - D2[t, R + r]
// and Im out[t, r] = D1[t, R + r] + D2[t, r].  The Laplace kernel needs D1 alone.
// G is formed on the CUDA cores in FP32 (rsqrt, sincos), both operands are split
// x = hi + lo into BF16, and three products (hi.hi + hi.lo + lo.hi, kind::f16,
// FP32 accumulation in TMEM) keep the product error near 2^-16; with more than 32
// right-hand sides lo.lo is added as well, which pays for the truncated additions
// there (kSegment).  With NP = 3 parts (hi + mid + lo, ~24 bits) six products take every
// p.q with p + q < 3, and the product error is near 2^-24.
//
// Why this shape.  G is the MMA's A operand and goes from registers straight into
// tensor memory: a thread owns one target (one TMEM lane), reads the entry's
// sources as broadcasts and forms 16 pairs per stage, so the per-stage hand-offs
// are paid once per 128 x 16 pairs, and no proxy fence or shared-memory tile is on
// the way.  The strengths are the B operand: one record per entry serves every
// target box of the unit.  (An earlier kernel had one target box per unit, T <= 32
// or 64 targets on the MMA's N side and both operands in shared memory: 3.7 M
// stages on the 2^21-point ellipsoid against 1.27 M entries here, every stage
// bound by its hand-offs; 64 right-hand sides there 5.15 ms per apply against 3.55,
// 24 in three parts on a 200 003-point sphere 676 us against 320.)
//
// Group records.  The B operand of a source group does not depend on the targets,
// so a pass per apply (k_tc_pack) writes every group's part images, already in the
// operand's shared-memory layout, followed by the group's source coordinates and
// markers of non-finite strengths; the main kernel moves a record with one TMA bulk
// copy.  Groups ignore box boundaries (n / 16 of them): which of the 16 sources a
// target meets is a 16-bit mask per (entry, target box).
//
// Lists (k_tc_fill, at plan time).  Blocks of 32 consecutive target boxes hold the
// union of their neighbour boxes' groups, ascending: the group, a bit per box of
// the block that has a neighbour source in it, and the boxes' 16-bit masks.  A
// block's targets are cut into near-equal windows of at most 128; a window takes
// the entries whose bits meet its own boxes.
//
// Main kernel (k_p2p_tc): persistent, one CTA per SM, units from a counter in
// Morton order (neighbouring CTAs share records in L2).  Warp roles:
//   warp 3       scout: takes units from the counter and reads their headers ahead of the producer
//   warp 0       producer: picks the unit's entries out of its block's list and issues entry e
//                into slot e % 16 (e % 8 where records are large): metadata, TMA bulk copies of the
//                record and of the masks
//   warps 1-2    MMA issuers (an elected lane each): D1 and D2 of every entry in order
//   warps 4-7    epilogue: TMEM -> a tile in shared memory, the complex combination, out[perm[t]]
//   warps 8-23   four G sets of four warps: entry e goes to set e % 4, which writes the BF16
//                parts of G into TMEM operand slot e % (operand slots)
// D occupies columns 0..255, the operand slots the other 256.  With at most 32
// right-hand sides the small products (all but hi.hi) have accumulators of their
// own.  The tensor core's FP32 accumulation truncates, ~2^-26 of the accumulator
// per MMA in the same direction, so chains are kept short: a unit's list is cut
// into near-equal segments (kSegment), and the epilogue adds the segments in
// FP32.
//
// Every wait is bounded: a wait that runs out sets the plan's status word and an
// abort flag; every role then stops, the producer waits (bounded) for the bulk
// copies it issued, each MMA issuer for its MMAs, and the CTA frees its TMEM and
// returns.
//
// The B operand uses the canonical K-major layout without swizzle: 8-row x 16-byte
// core matrices, the two K-adjacent cores of a 16-wide K slice 128 bytes apart
// (leading byte offset) and 8-row groups 256 bytes apart (stride byte offset).  A
// part of G is 8 TMEM columns, two consecutive sources per 32-bit column.
#include <math.h>

#include <algorithm>

#include "p2p_tc_common.cuh"

using namespace p2p_detail;
using namespace p2p_tc_common;

namespace {

constexpr int kImage = 2 * kPart;      // hi + lo images (the operand self-check)
constexpr int kRows = 128;             // targets per unit (MMA M)
constexpr int kBlockBoxes = 32;        // target boxes per list block (a bit each)
constexpr int kSets = 4;               // G sets; set s takes entries s, s + kSets, ...
// Entries added up in one accumulator chain at most.  With accumulators of their own for the small products (at most
// 32 right-hand sides) a chain takes one truncated addition per entry.  Wider launches have no TMEM left for that: every
// product of an entry is a truncated addition to the one accumulator, and with the three of hi / lo the error came out
// above that of the split alone even with short segments.  The fourth product, lo.lo, takes the split's own error from 4.4e-6
// to 3.5e-6, more than those additions cost, and the issuers have time for most of it (a G set takes ~750 cycles for an
// entry, its MMAs 384, 512 with the fourth).  Relative L2 error / time with 64 right-hand sides on 200 003 sphere points at 20 per box
// and on the 2^21-point ellipsoid, and with 40 at 47 points per box, entries per segment x products:
//   48 x 3  4.53e-6 331 us   5.00e-6 3556 us   4.64e-6
//   16 x 3  4.47e-6 401 us   5.06e-6 4340 us   4.50e-6
//   48 x 4  3.65e-6 346 us   3.70e-6 3673 us   3.86e-6
//   64 x 4  3.74e-6 332 us   3.80e-6 3546 us   3.93e-6; in a cube at 100 per box, where every slot of an entry is a pair,
//                                              4.98e-6 (one box per unit: 4.87e-6), at 75 per box 4.645e-6 (4.636e-6)
// (Six products per entry would need segments of 6 to 8 entries to be as exact as chains of ~55 additions, and the
// epilogue's share makes that slower than one box per unit: 2^21-point ellipsoid, 64 right-hand sides 7.4 ms against 6.9.
// p2p_tc_box.cu takes those calls.)
constexpr int kSegment = 48;
constexpr int kAColumn = 256;          // first TMEM column of the operand slots
constexpr int kMmaWarp0 = 1, kScoutWarp = 3, kEpiWarp0 = 4, kGWarp0 = 8;
constexpr int kWarps = kGWarp0 + 4 * kSets;
constexpr int kThreads = kWarps * 32;

// One poll without suspension.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Bounded wait; gives up early once *abort is set.  The first poll is the plain one: a barrier that has completed
// costs ~15 cycles with it, ~50 with the suspending one.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                          uint32_t limit = kWaitLimit) {
    if (limit > 0u && mbar_test(bar, parity)) return true;
    for (uint32_t i = 0; i < limit; ++i) {
        if (mbar_try(bar, parity)) return true;
        if (abort && (i & 15u) == 15u && *abort) return false;
    }
    return false;
}

// The A operand in tensor memory (128 lanes x 8 columns for K = 16).
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// One lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_lane() {
    uint32_t e;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(e));
    return e != 0;
}

// 32 lanes x 8 consecutive 32-bit columns of TMEM into registers; valid after tmem_ld_wait.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
// Orders the uses of v after every earlier load of this thread.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&v)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 :
                 : "memory");
}

// Registers into 4 consecutive 32-bit columns of the warp's 32 lanes; complete after tmem_st_wait.
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 lanes x 16 consecutive 32-bit columns of TMEM into registers.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Splits eight consecutive K elements (strengths) of one row into NP BF16 parts (2: hi, lo; 3: hi, mid, lo) stored at `off`
// in the images starting at part0, part_bytes apart.
template <int NP, bool CAP>
__device__ __forceinline__ void store_parts(unsigned char* part0, int part_bytes, int off, const float (&v)[8]) {
    uint32_t p[NP][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (NP == 2) split2<CAP>(v[2 * i], v[2 * i + 1], p[0][i], p[1][i]);
        else split3<CAP>(v[2 * i], v[2 * i + 1], p[0][i], p[1][i], p[2][i]);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q)
        *reinterpret_cast<uint4*>(part0 + q * part_bytes + off) = make_uint4(p[q][0], p[q][1], p[q][2], p[q][3]);
}

// ----------------------------------------------------------- strength pre-pack --

// Bytes of one group record for R = rhs (a multiple of 8) right-hand sides: NP part images of 2R rows x 16
// sources (rows 0..R-1 Re lambda, R..2R-1 Im lambda), the group's 16 x, y and z coordinates, four marker words
// (nonzero: some strength is not finite), and per source 64 bits naming its non-finite right-hand sides.
__host__ __device__ inline int image_bytes(int rhs) { return 2 * rhs * kSrcGroup * 2; }
constexpr int kXyzBytes = 3 * kSrcGroup * 4;
constexpr int kMarkBytes = 16;
constexpr int kBadBytes = kSrcGroup * 8;
// the part of a record the main kernel copies, and a record's size
__host__ __device__ inline int copy_bytes(int rhs, int np) { return np * image_bytes(rhs) + kXyzBytes + kMarkBytes; }
__host__ __device__ inline int record_bytes(int rhs, int np) { return (copy_bytes(rhs, np) + kBadBytes + 127) / 128 * 128; }

// Records of the groups of RHS [rhs0, rhs0 + rhs).  2 x RP threads per group (RP: rhs rounded up to whole warps):
// thread (o, r) splits Re and Im lambda of right-hand side rhs0 + r for sources 8o .. 8o + 7 into rows r and
// rhs + r of the part images.  Sources past the last one and RHS past nrhs are zero, and so is a strength that is
// not finite: its targets get their NaN in the main kernel's epilogue, since 0 x inf would reach the targets of
// the unit that are not its neighbours as well.  Memory bound: lambda is read once in full rows of up to 512
// bytes, the images written once.
template <int NP>
__global__ void __launch_bounds__(128) k_tc_pack(const float2* __restrict__ lam, int64_t ld, int32_t nrhs, int32_t rhs0,
                                                 int32_t rhs, const int32_t* __restrict__ perm,
                                                 const float4* __restrict__ xs, int64_t n, int32_t groups,
                                                 unsigned char* __restrict__ pack) {
    const int rp = (rhs + 31) & ~31;                        // 32 or 64
    const int tpg = 2 * rp;                                 // threads per group: 64 or 128
    const int sub = threadIdx.x / tpg, tid = threadIdx.x - sub * tpg;
    const int64_t g = (int64_t)blockIdx.x * (128 / tpg) + sub;
    if (g >= groups) return;
    const int o = tid / rp, r = tid - o * rp, lane = threadIdx.x & 31;
    const int64_t s0 = g * kSrcGroup + 8 * o;
    const int rr = rhs0 + r;
    unsigned char* rec = pack + g * record_bytes(rhs, NP);
    float re[8], im[8];
    uint32_t bad = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        float2 v = make_float2(0.f, 0.f);
        if (s0 + e < n && r < rhs && rr < nrhs) v = lam[(int64_t)perm[s0 + e] * ld + rr];
        const bool fin = isfinite(v.x) && isfinite(v.y);
        if (!fin) v = make_float2(0.f, 0.f);
        const uint32_t b = __ballot_sync(P2P_FULL_MASK, !fin);
        if (lane == e) bad = b;
        re[e] = v.x;
        im[e] = v.y;
    }
    if (r < rhs) {
        if (any_above(re) || any_above(im)) {
            store_parts<NP, true>(rec, image_bytes(rhs), op_off(r, 8 * o), re);
            store_parts<NP, true>(rec, image_bytes(rhs), op_off(rhs + r, 8 * o), im);
        } else {
            store_parts<NP, false>(rec, image_bytes(rhs), op_off(r, 8 * o), re);
            store_parts<NP, false>(rec, image_bytes(rhs), op_off(rhs + r, 8 * o), im);
        }
    }
    float* xyz = reinterpret_cast<float*>(rec + NP * image_bytes(rhs));
    uint32_t* mark = reinterpret_cast<uint32_t*>(rec + NP * image_bytes(rhs) + kXyzBytes);
    uint32_t* badw = mark + kMarkBytes / 4;
    const int w = r >> 5;                                   // 32-bit word of the 64 right-hand sides
    const uint32_t any = __ballot_sync(P2P_FULL_MASK, lane < 8 && bad != 0u);
    if (lane < 8) {
        badw[(8 * o + lane) * 2 + w] = bad;
        if (rp == 32) badw[(8 * o + lane) * 2 + 1] = 0u;
    }
    if (lane == 0) {
        mark[o * 2 + w] = any;
        if (rp == 32) mark[o * 2 + 1] = 0u;
    }
    if (w == 0 && lane < 8) {
        const float4 p = s0 + lane < n ? xs[s0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        xyz[8 * o + lane] = p.x;
        xyz[kSrcGroup + 8 * o + lane] = p.y;
        xyz[2 * kSrcGroup + 8 * o + lane] = p.z;
    }
}

// -------------------------------------------------------------------- list build --

// One warp per block of 32 target boxes (lane = box): an upper bound of its list (the groups that its boxes'
// neighbours cover, with repetitions), the number of its windows, and every target's box number in the block.
__global__ void __launch_bounds__(128) k_tc_blocks(const int32_t* __restrict__ box_ptr, int32_t nb,
                                                   const int32_t* __restrict__ src_box_ptr,
                                                   const int32_t* __restrict__ nbr_ptr,
                                                   const int32_t* __restrict__ nbr_idx, int32_t nblk,
                                                   int32_t* __restrict__ bound, int32_t* __restrict__ units,
                                                   uint8_t* __restrict__ member) {
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (j >= nblk) return;
    const int32_t b0 = (int32_t)j * kBlockBoxes, b1 = min(nb, b0 + kBlockBoxes);
    const int32_t b = b0 + lane;
    int s = 0;
    if (b < b1)
        for (int32_t e = nbr_ptr[b]; e < nbr_ptr[b + 1]; ++e) {
            const int32_t c = nbr_idx[e];
            s += (src_box_ptr[c + 1] - 1) / kSrcGroup - src_box_ptr[c] / kSrcGroup + 1;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(P2P_FULL_MASK, s, o);
    if (lane == 0) {
        bound[j] = s;
        units[j] = (box_ptr[b1] - box_ptr[b0] + kRows - 1) / kRows;
    }
    for (int32_t c = b0; c < b1; ++c)
        for (int32_t t = box_ptr[c] + lane; t < box_ptr[c + 1]; t += 32) member[t] = (uint8_t)(c - b0);
}

// One CTA per block: the sorted union of its boxes' neighbour boxes (at most 32 x 27, bitonic in shared memory),
// the groups they cover (ascending; neighbouring boxes may share one), and per group the boxes it concerns and
// their 16-bit source masks.  Also names the block of every one of its units.
constexpr int kFillThreads = 256;
constexpr int kUnionSlots = 1024;
static_assert(kBlockBoxes * 27 <= kUnionSlots, "a block's neighbour lists fit the sort buffer");
__global__ void __launch_bounds__(kFillThreads)
    k_tc_fill(const int32_t* __restrict__ src_box_ptr, const int32_t* __restrict__ nbr_ptr,
              const int32_t* __restrict__ nbr_idx, int32_t nb, const int32_t* __restrict__ off,
              const int32_t* __restrict__ ustart, int32_t* __restrict__ ecount, int32_t* __restrict__ unit_block,
              int32_t* __restrict__ gid, uint32_t* __restrict__ bits, uint32_t* __restrict__ masks) {
    __shared__ int32_t ub[kUnionSlots];    // sorted neighbour boxes, then the unique ones
    __shared__ int32_t pos[kUnionSlots];   // first entry of a unique box's own groups
    __shared__ int32_t first[kUnionSlots]; // the group at that entry
    __shared__ int32_t wsum[kFillThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t j = blockIdx.x;
    const int32_t b0 = j * kBlockBoxes, b1 = min(nb, b0 + kBlockBoxes);
    const int32_t e0 = nbr_ptr[b0], ne = nbr_ptr[b1] - e0;
    for (int32_t u = ustart[j] + tid; u < ustart[j + 1]; u += kFillThreads) unit_block[u] = j;
    for (int i = tid; i < kUnionSlots; i += kFillThreads) ub[i] = i < ne ? nbr_idx[e0 + i] : INT32_MAX;
    __syncthreads();
    for (int k = 2; k <= kUnionSlots; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            for (int i = tid; i < kUnionSlots; i += kFillThreads) {
                const int l = i ^ d;
                if (l > i) {
                    const int32_t x = ub[i], y = ub[l];
                    if (((i & k) == 0) ? x > y : x < y) {
                        ub[i] = y;
                        ub[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    // exclusive prefix over the threads of one value each; returns the prefix, `total` the sum
    auto block_scan = [&](int v, int& total) {
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(P2P_FULL_MASK, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kFillThreads / 32; ++w) {
            before += w < warp ? wsum[w] : 0;
            all += wsum[w];
        }
        __syncthreads();
        total = all;
        return before + x - v;
    };
    // unique boxes, compacted (kPer consecutive slots per thread)
    constexpr int kPer = kUnionSlots / kFillThreads;
    int32_t v[kPer];
    int cnt = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int p = tid * kPer + i;
        v[i] = ub[p];
        if (v[i] == INT32_MAX || (p > 0 && ub[p - 1] == v[i])) v[i] = -1;
        cnt += v[i] >= 0;
    }
    int nu;
    int at = block_scan(cnt, nu);  // its barriers also end every thread's reads of ub
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        if (v[i] >= 0) ub[at++] = v[i];
    __syncthreads();
    // own groups of every unique box: those its predecessor has not reached
    int lo_g[kPer], n_g[kPer];
    cnt = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int p = tid * kPer + i;
        lo_g[i] = n_g[i] = 0;
        if (p < nu) {
            const int32_t c = ub[p];
            lo_g[i] = src_box_ptr[c] / kSrcGroup;
            if (p > 0) lo_g[i] = max(lo_g[i], (src_box_ptr[ub[p - 1] + 1] - 1) / kSrcGroup + 1);
            n_g[i] = (src_box_ptr[c + 1] - 1) / kSrcGroup - lo_g[i] + 1;
        }
        cnt += n_g[i];
    }
    int total;
    at = block_scan(cnt, total);
    const int64_t base = off[j];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int p = tid * kPer + i;
        if (p < nu) {
            pos[p] = at;
            first[p] = lo_g[i];
            for (int q = 0; q < n_g[i]; ++q) gid[base + at + q] = lo_g[i] + q;
            at += n_g[i];
        }
    }
    if (tid == 0) ecount[j] = total;
    for (int i = tid; i < total; i += kFillThreads) bits[base + i] = 0u;
    for (int64_t i = tid; i < (int64_t)total * (kBlockBoxes / 2); i += kFillThreads) masks[base * (kBlockBoxes / 2) + i] = 0u;
    __syncthreads();
    // one warp per box of the block, lane = its neighbour: the sources of neighbour c in every group c reaches
    for (int32_t b = b0 + warp; b < b1; b += kFillThreads / 32) {
        const int32_t f0 = nbr_ptr[b], nn = nbr_ptr[b + 1] - f0;
        if (lane >= nn) continue;
        const int32_t c = nbr_idx[f0 + lane], m = b - b0;
        int lo = 0, hi = nu - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ub[mid] < c) lo = mid + 1;
            else hi = mid;
        }
        const int32_t sa = src_box_ptr[c], sb = src_box_ptr[c + 1];
        for (int32_t g = sa / kSrcGroup; g <= (sb - 1) / kSrcGroup; ++g) {
            const int64_t e = base + pos[lo] + (g - first[lo]);
            const int a = max(0, sa - g * kSrcGroup), z = min(kSrcGroup, sb - g * kSrcGroup);
            const uint32_t mk = ((1u << z) - 1u) & ~((1u << a) - 1u);
            atomicOr(masks + e * (kBlockBoxes / 2) + (m >> 1), mk << (16 * (m & 1)));
            atomicOr(bits + e, 1u << m);
        }
    }
}

// ------------------------------------------------------------------ main kernel --

struct TcArgs {
    const float4* xs;              // box-sorted target coordinates
    const unsigned char* pack;     // group records of this launch's right-hand sides
    const int32_t* off;            // per block: first entry
    const int32_t* ecount;         // per block: entries
    const int32_t* ustart;         // per block: first unit; [nblk]: units in all
    const int32_t* unit_block;     // per unit: its block
    const int32_t* gid;            // per entry: source group
    const uint32_t* bits;          // per entry: bit m = box m of the block has a neighbour source in it
    const uint16_t* masks;         // per entry and box of the block: which of the 16 sources are neighbours
    const uint8_t* member;         // per sorted target: box number in its block
    const int32_t* box_ptr;
    const int32_t* perm;
    // non-finite strengths only: the neighbour lists
    const int32_t* nbr_ptr;
    const int32_t* nbr_idx;
    const int32_t* src_box_ptr;
    float2* out;                   // first right-hand side of this launch
    int64_t ld;
    int32_t nrhs;                  // right-hand sides of this launch
    int32_t rhs;                   // the same rounded up to 8 (R)
    int32_t nb;
    int32_t nblk;
    int32_t slot_bytes;
    int32_t slots_log;             // log2 of the record slots (3 or 4)
    int32_t a_slots;               // TMEM operand slots (a power of two, at least kSets)
    int32_t vec_out;               // out and ld allow 16-byte stores
    float k;
    unsigned int* status;
    unsigned int* counter;         // [0] next unit, [1] CTAs done (both 0 between launches)
    uint32_t wait_limit;           // polls of every pipeline wait (kWaitLimit unless a self-check lowers it)
};

// Slot layout: the copied part of a record, the entry's masks, metadata.
constexpr int kMaskBytes = kBlockBoxes * 2;
__host__ __device__ inline int slot_xyz_off(int rhs, int np) { return np * image_bytes(rhs); }
__host__ __device__ inline int slot_mask_off(int rhs, int np) { return copy_bytes(rhs, np); }
__host__ __device__ inline int slot_meta_off(int rhs, int np) { return copy_bytes(rhs, np) + kMaskBytes; }
__host__ __device__ inline int slot_bytes_for(int rhs, int np) { return (slot_meta_off(rhs, np) + 16 + 127) / 128 * 128; }
constexpr int kMaxSlots = 16;
constexpr int kUnitQueue = 4;   // units the scout is ahead (a power of two)
// barriers, the epilogue's descriptor, the unit queue, TMEM address, abort flag
constexpr int kBarriers = 3 * kMaxSlots + 7 + 2 * kUnitQueue;
constexpr int kBarBytes = (16 + kUnitQueue * 32 + kBarriers * 8 + 8 + 127) / 128 * 128;
// The epilogue's tile: a row of 2R floats per target, padded so that 16-byte accesses of consecutive rows spread
// over the banks.
__host__ __device__ inline int tile_stride(int rhs) { return 2 * rhs + 4; }
__host__ __device__ inline int tile_bytes(int rhs) { return kRows * tile_stride(rhs) * 4; }
__host__ __device__ inline int tc_smem_bytes(int rhs, int np, int slots) {
    return slots * slot_bytes_for(rhs, np) + tile_bytes(rhs) + kBarBytes;
}

// Columns of an operand slot: NP parts of Gr and Gi, 8 columns each.
__host__ __device__ constexpr int a_cols(int np) { return np * 16; }

// Metadata of a stage (int4): x = flags, y = block's first box, z = the unit's first target, w = its targets.
// Flags: first / last entry of a segment, the end, a segment after the unit's first, the unit's last entry; in the
// epilogue's descriptor kFirst says that a strength of the segment is not finite.
constexpr int kFirst = 1, kLast = 2, kDone = 4, kAdd = 8, kOut = 16;

struct TcSmem {
    unsigned char* slots;
    float* tile;           // [kRows][tile_stride] sums of the epilogue
    uint64_t* full;        // [slots] TMA bytes + producer arrival
    uint64_t* full_a;      // [slots] one arrival per warp of the G set (operand slot written)
    uint64_t* done;        // [slots] MMA commits (record and operand slot free)
    uint64_t* desc_full;   // issuer 0: a finished segment's descriptor (or the end)
    uint64_t* acc_full;    // [2] an issuer's commit after a segment's last entry
    uint64_t* acc_empty;   // [2] the epilogue's warps have read D1, D2
    uint64_t* drain;       // [2] an issuer's MMAs after an abort
    uint64_t* uq_full;     // [kUnitQueue] scout -> producer
    uint64_t* uq_empty;    // [kUnitQueue] producer -> scout
    int4* desc;
    int4* uq;              // [2 kUnitQueue] unit headers
    uint32_t* tmem_slot;
    int* abort;
    uint32_t mask, log;    // slots - 1, log2 of the slots
    // Entry numbers run over all units of the CTA: entry e uses record slot e % slots in its (e / slots)-th round.
    __device__ __forceinline__ uint32_t slot(uint32_t e) const { return e & mask; }
    __device__ __forceinline__ uint32_t phase(uint32_t e) const { return (e >> log) & 1u; }
};

__device__ __forceinline__ TcSmem carve(unsigned char* smem, const TcArgs& a) {
    TcSmem s;
    s.log = (uint32_t)a.slots_log;
    s.mask = (1u << s.log) - 1u;
    s.slots = smem;
    unsigned char* p = smem + ((size_t)a.slot_bytes << s.log);
    s.tile = reinterpret_cast<float*>(p);
    p += tile_bytes(a.rhs);
    s.desc = reinterpret_cast<int4*>(p);
    s.uq = s.desc + 1;
    uint64_t* b = reinterpret_cast<uint64_t*>(p + 16 + kUnitQueue * 32);
    s.full = b;
    s.full_a = b + kMaxSlots;
    s.done = b + 2 * kMaxSlots;
    s.desc_full = b + 3 * kMaxSlots;
    s.acc_full = b + 3 * kMaxSlots + 1;
    s.acc_empty = b + 3 * kMaxSlots + 3;
    s.drain = b + 3 * kMaxSlots + 5;
    s.uq_full = b + 3 * kMaxSlots + 7;
    s.uq_empty = s.uq_full + kUnitQueue;
    s.tmem_slot = reinterpret_cast<uint32_t*>(b + kBarriers);
    s.abort = reinterpret_cast<int*>(s.tmem_slot + 1);
    return s;
}

__device__ __forceinline__ void set_abort(const TcArgs& a, const TcSmem& sm) {
    *(volatile int*)sm.abort = 1;
    atomicOr(a.status, P2P_DEV_TIMEOUT | P2P_DEV_TC_FAULTED);
}

// Wait of a whole warp: every lane polls, and all lanes get the same answer.
__device__ __forceinline__ bool warp_wait(const TcArgs& a, const TcSmem& sm, uint64_t* bar, uint32_t parity,
                                          uint32_t limit) {
    const bool ok = mbar_wait(bar, parity, sm.abort, limit);
    if (__all_sync(P2P_FULL_MASK, ok)) return true;
    if (!ok && !*(volatile int*)sm.abort) set_abort(a, sm);
    return false;
}

// ---- scout (one warp) ----
// Unit headers: (block's first box, first target, targets, entries), (first list entry, list length, the window's
// boxes as bits, entries per segment).  Its chain of dependent loads takes several microseconds a unit, which the
// queue hides.  Zero entries end the queue.
template <bool LIMITED, int NP>
__device__ void run_scout(const TcArgs& a, const TcSmem& sm, int lane) {
    const uint32_t wlim = LIMITED ? a.wait_limit : kWaitLimit;
    const int units = a.ustart[a.nblk];
    auto next_unit = [&]() { return lane == 0 ? (int)atomicAdd(a.counter, 1u) : 0; };
    uint32_t at = 0;
    int un = next_unit();
    while (true) {
        const int u = __shfl_sync(P2P_FULL_MASK, un, 0);
        int4 h0 = make_int4(0, 0, 0, 0), h1 = h0;
        if (u < units) {
            un = next_unit();
            const int j = a.unit_block[u];
            const int b0 = j * kBlockBoxes;
            const int p0 = a.box_ptr[b0], p1 = a.box_ptr[min(a.nb, b0 + kBlockBoxes)];
            const int off = a.off[j], E = a.ecount[j], first = a.ustart[j], windows = a.ustart[j + 1] - first;
            const int size = (p1 - p0 + windows - 1) / windows;
            const int t0 = p0 + (u - first) * size;
            const int nt = min(size, p1 - t0);
            if (nt <= 0) continue;
            const int m0 = a.member[t0], m1 = a.member[t0 + nt - 1];
            const uint32_t want = (0xffffffffu << m0) & (0xffffffffu >> (31 - m1));
            int cnt = 0;
#pragma unroll 4
            for (int i = lane; i < E; i += 32) cnt += (a.bits[(int64_t)off + i] & want) != 0u;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(P2P_FULL_MASK, cnt, o);
            if (cnt == 0) continue;  // two point sets, no source nearby: the rows keep the zeros written before the launch
            const int segments = (cnt + kSegment - 1) / kSegment;
            h0 = make_int4(b0, t0, nt, cnt);
            h1 = make_int4(off, E, (int)want, (cnt + segments - 1) / segments);
        }
        const uint32_t q = at & (uint32_t)(kUnitQueue - 1), ph = (at / kUnitQueue) & 1u;
        if (!warp_wait(a, sm, &sm.uq_empty[q], ph ^ 1u, wlim)) return;
        if (lane == 0) {
            sm.uq[2 * q] = h0;
            sm.uq[2 * q + 1] = h1;
            mbar_arrive(&sm.uq_full[q]);
        }
        __syncwarp();
        if (h0.w == 0) return;
        ++at;
    }
}

// ---- producer (one warp) ----
// Up to kBatch entries at a time, a lane each: the polls, the fence and the barrier operations of a batch overlap
// (one lane issuing entry by entry took ~1 000 cycles per entry).
constexpr int kBatch = 2;
template <bool LIMITED, int NP>
__device__ void run_producer(const TcArgs& a, const TcSmem& sm, int lane) {
    const uint32_t wlim = LIMITED ? a.wait_limit : kWaitLimit;
    const uint32_t copy = (uint32_t)copy_bytes(a.rhs, NP);
    const int64_t rec = record_bytes(a.rhs, NP);
    const int mask_off = slot_mask_off(a.rhs, NP), meta_off = slot_meta_off(a.rhs, NP);
    // entry ee's slot is free (lanes with `mine`)
    auto claim = [&](bool mine, uint32_t ee) {
        bool ok = true;
        if (mine) ok = mbar_wait(&sm.done[sm.slot(ee)], sm.phase(ee) ^ 1u, sm.abort, wlim);
        if (__all_sync(P2P_FULL_MASK, ok)) return true;
        if (!ok && !*(volatile int*)sm.abort) set_abort(a, sm);
        return false;
    };
    uint32_t e = 0, armed = 0;  // entries numbered; entries whose copies may still be in flight
    bool failed = false;
    for (uint32_t at = 0; !failed; ++at) {
        const uint32_t q = at & (uint32_t)(kUnitQueue - 1);
        if (!warp_wait(a, sm, &sm.uq_full[q], (at / kUnitQueue) & 1u, wlim)) {
            failed = true;
            break;
        }
        const int4 h0 = sm.uq[2 * q], h1 = sm.uq[2 * q + 1];
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.uq_empty[q]);
        const int b0 = h0.x, t0 = h0.y, nt = h0.z, cnt = h0.w, E = h1.y, len = h1.w;
        if (cnt == 0) break;
        const int64_t off = h1.x;
        const uint32_t want = (uint32_t)h1.z;
        int k = 0;  // entries of the unit so far
        uint32_t bt = lane < E ? a.bits[off + lane] : 0u;
        int g = lane < E ? a.gid[off + lane] : 0;
        for (int w0 = 0; w0 < E && !failed; w0 += 32) {
            const bool valid = (bt & want) != 0u;
            const int gs = g;
            const bool in = w0 + 32 + lane < E;  // the next 32 entries, in flight
            bt = in ? a.bits[off + w0 + 32 + lane] : 0u;
            g = in ? a.gid[off + w0 + 32 + lane] : 0;
            const uint32_t todo = __ballot_sync(P2P_FULL_MASK, valid);
            const int rank = __popc(todo & ((1u << lane) - 1u)), n = __popc(todo);
            const uint32_t ee = e + (uint32_t)rank;
            const int kk = k + rank, in_seg = kk % len;
            const int flags = (in_seg == 0 ? kFirst : 0) | (in_seg == len - 1 || kk == cnt - 1 ? kLast : 0) |
                              (kk >= len ? kAdd : 0) | (kk == cnt - 1 ? kOut : 0);
            for (int i0 = 0; i0 < n; i0 += kBatch) {
                const bool mine = valid && rank >= i0 && rank < i0 + kBatch;
                if (!claim(mine, ee)) {
                    failed = true;
                    break;
                }
                if (mine) {
                    unsigned char* base = sm.slots + (size_t)sm.slot(ee) * a.slot_bytes;
                    uint64_t* bar = &sm.full[sm.slot(ee)];
                    *reinterpret_cast<int4*>(base + meta_off) = make_int4(flags, b0, t0, nt);
                    fence_async_smem();  // the slot was last read through the generic proxy
                    mbar_expect_tx(bar, copy + (uint32_t)kMaskBytes);
                    bulk_g2s(base, a.pack + gs * rec, copy, bar);
                    bulk_g2s(base + mask_off, a.masks + (off + w0 + lane) * kBlockBoxes, (uint32_t)kMaskBytes, bar);
                }
                __syncwarp();
                armed = e + (uint32_t)min(n, i0 + kBatch);
            }
            e += (uint32_t)n;
            k += n;
        }
    }
    // a terminal stage for every G set (the issuers stop at the first)
    if (!failed) {
        const bool mine = lane < kSets;
        const uint32_t ee = e + (uint32_t)lane;
        failed = !claim(mine, ee);
        if (!failed && mine) {
            *reinterpret_cast<int4*>(sm.slots + (size_t)sm.slot(ee) * a.slot_bytes + meta_off) = make_int4(kDone, 0, -1, 0);
            mbar_arrive(&sm.full[sm.slot(ee)]);
        }
    }
    if (failed && lane == 0)  // wait (bounded) for the copies of the latest round of slots
        for (uint32_t i = armed > sm.mask + 1u ? armed - sm.mask - 1u : 0u; i < armed; ++i)
            mbar_wait(&sm.full[sm.slot(i)], sm.phase(i), nullptr, kDrainLimit);
}

// ---- G sets (128 threads each: thread = target = TMEM lane) ----
// G of target t (negated coordinates ntx, nty, ntz) against sources 8H .. 8H + 7 of the entry, those of `mask`:
// NP BF16 parts of Re and Im, two sources per word.  The sources go in pairs through the packed two-lane FP32
// instructions; rsqrt and sincos stay per pair.  r = 0 and sources outside the mask give 0 (whatever their
// distance evaluates to).
template <int KERN, int NP, int H>
__device__ __forceinline__ void g_eight(const float* __restrict__ xyz, float2 ntx, float2 nty, float2 ntz, float2 k2,
                                        uint32_t mask, uint32_t (&re)[NP][4], uint32_t (&im)[NP][4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float4 X = *reinterpret_cast<const float4*>(xyz + 8 * H + 4 * q);
        const float4 Y = *reinterpret_cast<const float4*>(xyz + kSrcGroup + 8 * H + 4 * q);
        const float4 Z = *reinterpret_cast<const float4*>(xyz + 2 * kSrcGroup + 8 * H + 4 * q);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int s = 8 * H + 4 * q + 2 * c, w = 2 * q + c;
            const float2 dx = __fadd2_rn(c ? make_float2(X.z, X.w) : make_float2(X.x, X.y), ntx);
            const float2 dy = __fadd2_rn(c ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y), nty);
            const float2 dz = __fadd2_rn(c ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y), ntz);
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            const float2 inv = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            const bool ok0 = r2.x > 0.f && ((mask >> s) & 1u), ok1 = r2.y > 0.f && ((mask >> (s + 1)) & 1u);
            float2 gr = inv, gi = make_float2(0.f, 0.f);
            if (KERN == P2P_HELMHOLTZ) {
                const float2 ph = __fmul2_rn(k2, __fmul2_rn(r2, inv));
                float2 sn, cs;
                __sincosf(ph.x, &sn.x, &cs.x);
                __sincosf(ph.y, &sn.y, &cs.y);
                gr = __fmul2_rn(cs, inv);
                gi = __fmul2_rn(sn, inv);
            }
            const float r0 = ok0 ? gr.x : 0.f, r1 = ok1 ? gr.y : 0.f;
            if constexpr (NP == 2) split2(r0, r1, re[0][w], re[1][w]);
            else split3(r0, r1, re[0][w], re[1][w], re[2][w]);
            if (KERN == P2P_HELMHOLTZ) {
                const float i0 = ok0 ? gi.x : 0.f, i1 = ok1 ? gi.y : 0.f;
                if constexpr (NP == 2) split2(i0, i1, im[0][w], im[1][w]);
                else split3(i0, i1, im[0][w], im[1][w], im[2][w]);
            }
        }
    }
}

// The eight sources' parts into operand slot `col`: part p of Re at columns 16p + 4H.., of Im 8 further.
template <int KERN, int NP, int H>
__device__ __forceinline__ void store_eight(uint32_t col, const uint32_t (&re)[NP][4], const uint32_t (&im)[NP][4]) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        tmem_st4(col + 16 * p + 4 * H, re[p][0], re[p][1], re[p][2], re[p][3]);
        if (KERN == P2P_HELMHOLTZ) tmem_st4(col + 16 * p + 8 + 4 * H, im[p][0], im[p][1], im[p][2], im[p][3]);
    }
}

template <int KERN, bool LIMITED, int NP>
__device__ void run_gset(const TcArgs& a, const TcSmem& sm, uint32_t tmem, int set, int quadrant, int lane) {
    const uint32_t wlim = LIMITED ? a.wait_limit : kWaitLimit;
    const int xyz_off = slot_xyz_off(a.rhs, NP), mask_off = slot_mask_off(a.rhs, NP), meta_off = slot_meta_off(a.rhs, NP);
    const int row = quadrant * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quadrant * 32) << 16) + (uint32_t)kAColumn;
    const float2 k2 = make_float2(a.k, a.k);
    float2 ntx = make_float2(0.f, 0.f), nty = ntx, ntz = ntx;
    int unit = -1, m = -1;  // first target of the current unit, this target's box number (-1: no target)
    for (uint32_t e = (uint32_t)set;; e += kSets) {
        unsigned char* base = sm.slots + (size_t)sm.slot(e) * a.slot_bytes;
        if (!warp_wait(a, sm, &sm.full[sm.slot(e)], sm.phase(e), wlim)) break;
        const int4 meta = *reinterpret_cast<const int4*>(base + meta_off);
        if (meta.x & kDone) {
            if (lane == 0) mbar_arrive(&sm.full_a[sm.slot(e)]);
            break;
        }
        if (meta.z != unit) {
            unit = meta.z;
            m = -1;
            if (row < meta.w) {
                const float4 t = a.xs[unit + row];
                m = a.member[unit + row];
                ntx = make_float2(-t.x, -t.x);
                nty = make_float2(-t.y, -t.y);
                ntz = make_float2(-t.z, -t.z);
            }
        }
        const uint32_t mask = m >= 0 ? reinterpret_cast<const uint16_t*>(base + mask_off)[m] : 0u;
        const float* xyz = reinterpret_cast<const float*>(base + xyz_off);
        const uint32_t col = lane_addr + (e & (uint32_t)(a.a_slots - 1)) * (uint32_t)a_cols(NP);
        // halves of the group that hold a source near one of the warp's targets
        const uint32_t some = __reduce_or_sync(P2P_FULL_MASK, mask);
        const bool any0 = (some & 0xffu) != 0u, any1 = some > 0xffu;
        uint32_t re[NP][4], im[NP][4];
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int w = 0; w < 4; ++w) re[p][w] = im[p][w] = 0u;
        if (any0) g_eight<KERN, NP, 0>(xyz, ntx, nty, ntz, k2, mask, re, im);
        // the operand slot is free: the MMAs of entry e - a_slots are done
        if (e >= (uint32_t)a.a_slots) {
            const uint32_t p = e - (uint32_t)a.a_slots;
            if (!warp_wait(a, sm, &sm.done[sm.slot(p)], sm.phase(p), wlim)) break;
            tc_fence_after();
        }
        store_eight<KERN, NP, 0>(col, re, im);
        if (any1) {
            g_eight<KERN, NP, 1>(xyz, ntx, nty, ntz, k2, mask, re, im);
        } else if (any0) {
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int w = 0; w < 4; ++w) re[p][w] = im[p][w] = 0u;
        }
        store_eight<KERN, NP, 1>(col, re, im);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.full_a[sm.slot(e)]);
    }
}

// ---- MMA issuer Q (one warp, an elected lane): Q = 0 adds Gr [Lr | Li] into D1, Q = 1 Gi [Lr | Li] into D2 ----
template <bool LIMITED, int NP>
__device__ void run_mma(const TcArgs& a, const TcSmem& sm, uint32_t tmem, int q) {
    const uint32_t wlim = LIMITED ? a.wait_limit : kWaitLimit;
    const int meta_off = slot_meta_off(a.rhs, NP), mark_off = slot_xyz_off(a.rhs, NP) + kXyzBytes;
    const uint32_t idesc = idesc_bf16_f32(2 * a.rhs);
    // a descriptor's start address is its low 14 bits, in 16-byte units: a slot adds its offset, a part its own
    // (shared memory stays below 2^18 bytes, so the sums never carry out of the field)
    const uint64_t db_all = smem_desc(smem_u32(sm.slots));
    const uint32_t slot16 = (uint32_t)a.slot_bytes >> 4;
    const uint64_t part = (uint64_t)(image_bytes(a.rhs) >> 4);
    const uint32_t d_hh = tmem + (uint32_t)q * 128u;                 // hi.hi
    const uint32_t d_x = a.rhs <= 32 ? d_hh + 64u : d_hh;            // the smaller products
    const uint32_t one_x = a.rhs <= 32 ? 0u : 1u;                    // 1: they share the accumulator of hi.hi
    const uint32_t ga_all = tmem + (uint32_t)kAColumn + 8u * (uint32_t)q, a_mask = (uint32_t)(a.a_slots - 1);
    const int lane = threadIdx.x & 31;
    // The products of one entry (the elected lane): every product of parts p (of G) and r (of lambda) with
    // p + r < NP, and lo.lo of a wide hi / lo launch; the dropped ones are below 2^-8 NP of the leading one.
    auto issue = [&](uint32_t ga, uint64_t lb, uint32_t acc, uint64_t* done) {
        mma_bf16_ts(d_hh, ga, lb, idesc, acc);
        mma_bf16_ts(d_x, ga, lb + part, idesc, acc | one_x);
        mma_bf16_ts(d_x, ga + 16u, lb, idesc, 1u);
        if constexpr (NP == 2) {
            if (one_x) mma_bf16_ts(d_x, ga + 16u, lb + part, idesc, 1u);
        } else {
            mma_bf16_ts(d_x, ga, lb + 2 * part, idesc, 1u);
            mma_bf16_ts(d_x, ga + 16u, lb + part, idesc, 1u);
            mma_bf16_ts(d_x, ga + 32u, lb, idesc, 1u);
        }
        mma_commit(done);
    };
    // Several entries at a time: lane i polls the barriers and reads the metadata of entry e + i.  (Entry by entry,
    // the polls and the metadata of an entry took this warp ~600 cycles, the MMAs ~200.)  Half of the operand
    // slots, so that the G sets fill the other half meanwhile.
    constexpr int kTake = NP == 2 ? 4 : 2;
    uint32_t seg = 0, acc = 0u;  // acc 0: the segment's first entry
    bool bad = false, ended = false, ok = true, issued = false;
    int4 meta = make_int4(0, 0, 0, 0);  // lane i: entry e + i
    uint32_t special = 0u, marks = 0u;  // bit i: entry e + i starts or ends something; has a strength that is not finite
    // lanes 0 .. 3 poll the operand slots, lanes 4 .. 7 the records (complete by then: the G set waited for them)
    auto bar_of = [&](uint32_t le) { return (lane & 4) ? &sm.full[sm.slot(le)] : &sm.full_a[sm.slot(le)]; };
    auto read_batch = [&](uint32_t le) {
        const unsigned char* base = sm.slots + (size_t)sm.slot(le) * a.slot_bytes;
        meta = *reinterpret_cast<const int4*>(base + meta_off);
        const int4 mk = *reinterpret_cast<const int4*>(base + mark_off);
        special = __ballot_sync(P2P_FULL_MASK, (meta.x & (kFirst | kLast | kDone)) != 0);
        marks = __ballot_sync(P2P_FULL_MASK, !(meta.x & kDone) && (mk.x | mk.y | mk.z | mk.w) != 0);
        tc_fence_after();
    };
    bool ready = false;  // the batch at e has been polled and read
    for (uint32_t e = 0; ok && !ended; e += kTake) {
        const uint32_t le = e + (uint32_t)(lane & (kTake - 1));
        if (!ready) {
            if (!warp_wait(a, sm, bar_of(le), sm.phase(le), wlim)) break;
            read_batch(le);
        }
        ready = false;
        const uint32_t ga0 = ga_all + (e & a_mask) * (uint32_t)a_cols(NP);
        const uint64_t lb0 = db_all + (uint64_t)(sm.slot(e) * slot16);
        uint64_t* done0 = &sm.done[sm.slot(e)];
        issued = true;
        if (special == 0u) {
            // inside a segment: the next batch is polled between the two halves, while the first one's MMAs run
            bad |= marks != 0u;
            if (elect_lane()) {
#pragma unroll
                for (int i = 0; i < kTake / 2; ++i)
                    issue(ga0 + (uint32_t)(i * a_cols(NP)), lb0 + (uint64_t)(i * slot16), 1u, done0 + i);
            }
            __syncwarp();
            const uint32_t ne = le + kTake;
            ready = __all_sync(P2P_FULL_MASK, mbar_test(bar_of(ne), sm.phase(ne)));
            if (ready) read_batch(ne);
            if (elect_lane()) {
#pragma unroll
                for (int i = kTake / 2; i < kTake; ++i)
                    issue(ga0 + (uint32_t)(i * a_cols(NP)), lb0 + (uint64_t)(i * slot16), 1u, done0 + i);
            }
            __syncwarp();
            continue;
        }
        for (int i = 0; i < kTake; ++i) {
            const int flags = __shfl_sync(P2P_FULL_MASK, meta.x, i);
            if (flags & (kFirst | kDone)) {
                // the epilogue has read this issuer's accumulator (and the descriptor) of the segment before
                if (!warp_wait(a, sm, &sm.acc_empty[q], (seg & 1u) ^ 1u, wlim)) {
                    ok = false;
                    break;
                }
                if (flags & kDone) {
                    ended = true;
                    break;
                }
                acc = 0u;
                bad = false;
            }
            bad |= ((marks >> i) & 1u) != 0;
            if (elect_lane()) {
                issue(ga0 + (uint32_t)(i * a_cols(NP)), lb0 + (uint64_t)(i * slot16), acc, done0 + i);
                if (flags & kLast) mma_commit(&sm.acc_full[q]);
            }
            acc = 1u;
            if (flags & kLast) {
                if (q == 0 && lane == i) {  // this entry's metadata is lane i's
                    *sm.desc = make_int4((flags & (kAdd | kOut)) | (bad ? kFirst : 0), meta.y, meta.z, meta.w);
                    mbar_arrive(sm.desc_full);
                }
                ++seg;
            }
            __syncwarp();
        }
    }
    if (elect_lane()) {
        if (ended && q == 0) {
            *sm.desc = make_int4(kDone, 0, 0, 0);
            mbar_arrive(sm.desc_full);
        } else if (!ended && issued) {
            // this warp's MMAs in flight
            mma_commit(&sm.drain[q]);
            mbar_wait(&sm.drain[q], 0u, nullptr, kDrainLimit);
        }
    }
    __syncwarp();
}

// Right-hand sides for which some source near sorted target t has a non-finite strength (bit r).
template <int NP>
__device__ __noinline__ uint64_t bad_rhs(const TcArgs& a, int t, int b0) {
    const int64_t rec = record_bytes(a.rhs, NP);
    const int b = b0 + a.member[t];
    uint64_t bad = 0;
    for (int e = a.nbr_ptr[b]; e < a.nbr_ptr[b + 1]; ++e) {
        const int c = a.nbr_idx[e];
        for (int s = a.src_box_ptr[c]; s < a.src_box_ptr[c + 1]; ++s) {
            const uint32_t* w = reinterpret_cast<const uint32_t*>(a.pack + (s / kSrcGroup) * rec + copy_bytes(a.rhs, NP)) +
                                2 * (s % kSrcGroup);
            bad |= (uint64_t)w[0] | ((uint64_t)w[1] << 32);
        }
    }
    return bad;
}

// ---- epilogue (four warps, each its own quadrant of TMEM lanes: lane = target) ----
// A segment's accumulators go through registers into the tile in shared memory, added up over the unit's segments in
// FP32: first D1, which the first issuer may then overwrite, then D2.  Finished rows leave from the tile while the
// next segment's MMAs run.  (Rows stored from the registers, 16 bytes per target and instruction, held the
// accumulators for ~16 000 cycles.)
template <int KERN, bool LIMITED, int NP>
__device__ void run_epilogue(const TcArgs& a, const TcSmem& sm, uint32_t tmem, int quadrant, int lane) {
    const uint32_t wlim = LIMITED ? a.wait_limit : kWaitLimit;
    const uint32_t lane_addr = tmem + ((uint32_t)(quadrant * 32) << 16);
    const int row = quadrant * 32 + lane;
    const int stride = tile_stride(a.rhs);
    const bool split = a.rhs <= 32;
    float* mine = sm.tile + row * stride;
    // columns of right-hand sides r0 .. r0 + 7 in accumulator q: x those of Lr, y those of Li
    auto load = [&](int q, int r0, float2 (&x)[4], float2 (&y)[4]) {
        uint32_t u[8], v[8], s[8], t[8];
        const uint32_t col = lane_addr + 128u * (uint32_t)q + (uint32_t)r0;
        tmem_ld8(col, u);
        tmem_ld8(col + (uint32_t)a.rhs, v);
        if (split) {
            tmem_ld8(col + 64u, s);
            tmem_ld8(col + 64u + (uint32_t)a.rhs, t);
        }
        tmem_ld_wait(u);
        tmem_ld_wait(v);
        if (split) {
            tmem_ld_wait(s);
            tmem_ld_wait(t);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[i] = make_float2(__uint_as_float(u[2 * i]), __uint_as_float(u[2 * i + 1]));
            y[i] = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            if (split) {
                x[i] = __fadd2_rn(x[i], make_float2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])));
                y[i] = __fadd2_rn(y[i], make_float2(__uint_as_float(t[2 * i]), __uint_as_float(t[2 * i + 1])));
            }
        }
    };
    for (uint32_t seg = 0;; ++seg) {
        if (!warp_wait(a, sm, sm.desc_full, seg & 1u, wlim)) return;
        const int4 d = *sm.desc;
        if (d.x & kDone) return;
        const bool valid = row < d.w;
        const int32_t out_row = valid ? a.perm[d.z + row] : 0;
        uint64_t bad = 0;
        if ((d.x & kFirst) && valid) bad = bad_rhs<NP>(a, d.z + row, d.y);
        if (!warp_wait(a, sm, &sm.acc_full[0], seg & 1u, wlim)) return;
        tc_fence_after();
        for (int r0 = 0; r0 < a.rhs; r0 += 8) {
            float2 x[4], y[4];
            load(0, r0, x, y);
            if (bad) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float nan = __int_as_float(0x7fc00000);
                    if ((bad >> (r0 + 2 * i)) & 1u) x[i].x = y[i].x = nan;
                    if ((bad >> (r0 + 2 * i + 1)) & 1u) x[i].y = y[i].y = nan;
                }
            }
            float4* to = reinterpret_cast<float4*>(mine + 2 * r0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 w = make_float4(x[i].x, y[i].x, x[i].y, y[i].y);
                if (d.x & kAdd) {
                    const float4 o = to[i];
                    w = make_float4(w.x + o.x, w.y + o.y, w.z + o.z, w.w + o.w);
                }
                to[i] = w;
            }
        }
        // D1's columns are in shared memory, and the descriptor in registers
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.acc_empty[0]);
        if (KERN == P2P_HELMHOLTZ) {
            if (!warp_wait(a, sm, &sm.acc_full[1], seg & 1u, wlim)) return;
            tc_fence_after();
            for (int r0 = 0; r0 < a.rhs; r0 += 8) {
                float2 x[4], y[4];
                load(1, r0, x, y);
                float4* to = reinterpret_cast<float4*>(mine + 2 * r0);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 o = to[i];
                    to[i] = make_float4(o.x - y[i].x, o.y + x[i].x, o.z - y[i].y, o.w + x[i].y);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.acc_empty[1]);
        }
        if (d.x & kOut) {
            // eight rows at a time, four lanes for a row's 64 bytes
            const int piece = 2 * (lane & 3);
            for (int i = 0; i < 32; i += 8) {
                const int rr = i + (lane >> 2);
                float2* dst = a.out + (int64_t)__shfl_sync(P2P_FULL_MASK, out_row, rr) * a.ld;
                if (quadrant * 32 + rr >= d.w) continue;
                for (int r = piece; r < a.nrhs; r += 8) {
                    const float4 w = *reinterpret_cast<const float4*>(sm.tile + (quadrant * 32 + rr) * stride + 2 * r);
                    const float2 w0 = make_float2(w.x * kInv4Pi, w.y * kInv4Pi), w1 = make_float2(w.z * kInv4Pi, w.w * kInv4Pi);
                    if (a.vec_out && r + 1 < a.nrhs) {
                        *reinterpret_cast<float4*>(dst + r) = make_float4(w0.x, w0.y, w1.x, w1.y);
                    } else {
                        dst[r] = w0;
                        if (r + 1 < a.nrhs) dst[r + 1] = w1;
                    }
                }
            }
            __syncwarp();  // the rows are read before the next segment overwrites them
        }
    }
}

// LIMITED: the waits poll at most a.wait_limit times (the abort-path self-check); otherwise kWaitLimit.
// NP: BF16 parts per operand (2: three or four products per entry and chain, 3: six).
template <int KERN, bool LIMITED, int NP>
__global__ void __launch_bounds__(kThreads, 1) k_p2p_tc(const __grid_constant__ TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const TcSmem sm = carve(smem, a);
    constexpr int kIssuers = KERN == P2P_HELMHOLTZ ? 2 : 1;
    if (warp == 0) tmem_alloc(sm.tmem_slot, 512u);
    if (tid == 32) {
        for (int i = 0; i < 1 << a.slots_log; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.full_a[i], 4);
            mbar_init(&sm.done[i], kIssuers);
        }
        mbar_init(sm.desc_full, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.acc_full[i], 1);
            mbar_init(&sm.acc_empty[i], 4);
        }
        for (int i = 0; i < kUnitQueue; ++i) {
            mbar_init(&sm.uq_full[i], 1);
            mbar_init(&sm.uq_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) mbar_init(&sm.drain[i], 1);
        *sm.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *sm.tmem_slot;
    if (warp == 0) {
        run_producer<LIMITED, NP>(a, sm, lane);
    } else if (warp < kMmaWarp0 + kIssuers) {
        run_mma<LIMITED, NP>(a, sm, tmem, warp - kMmaWarp0);
    } else if (warp == kScoutWarp) {
        run_scout<LIMITED, NP>(a, sm, lane);
    } else if (warp >= kGWarp0) {
        run_gset<KERN, LIMITED, NP>(a, sm, tmem, (warp - kGWarp0) >> 2, warp & 3, lane);
    } else if (warp >= kEpiWarp0) {
        run_epilogue<KERN, LIMITED, NP>(a, sm, tmem, warp & 3, lane);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512u);
    }
    // the last CTA leaves the unit counter at zero for the next launch
    if (tid == kScoutWarp * 32) {
        __threadfence();
        if (atomicAdd(a.counter + 1, 1u) == gridDim.x - 1u) {
            a.counter[0] = 0u;
            a.counter[1] = 0u;
        }
    }
}

// ------------------------------------------------- operand-layout self-check --

// D[128 x N] = A[128 x K] . B[N x K]^T with A, B split into BF16 hi + lo (3 MMAs
// per 16-wide K slice), both operands in shared memory, through the operand layout,
// descriptors and instruction descriptor of k_p2p_tc's B operand.
__global__ void __launch_bounds__(128, 1) k_tc_gemm_check(const float* __restrict__ A, const float* __restrict__ B,
                                                          float* __restrict__ D, int K, int n, int tmem_cols,
                                                          unsigned int* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* a_hi = smem;
    unsigned char* a_lo = a_hi + kImage / 2;
    unsigned char* b_hi = smem + kImage;
    unsigned char* b_lo = b_hi + (n / 8) * kSbo;
    uint64_t* bar = reinterpret_cast<uint64_t*>(b_lo + (n / 8) * kSbo);
    uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 1);
    if (warp == 0) tmem_alloc(slot, (uint32_t)tmem_cols);
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    const uint32_t idesc = idesc_bf16_f32(n);
    bool ok = true;
    for (int ks = 0; ks < K / kSrcGroup && ok; ++ks) {
        for (int c = tid; c < 128 * 2; c += 128) {
            const int row = c >> 1, half = c & 1;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = A[(int64_t)row * K + ks * 16 + half * 8 + i];
            store_parts<2, false>(a_hi, (int)(a_lo - a_hi), op_off(row, half * 8), v);
        }
        for (int c = tid; c < n * 2; c += 128) {
            const int row = c >> 1, half = c & 1;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = B[(int64_t)row * K + ks * 16 + half * 8 + i];
            store_parts<2, false>(b_hi, (int)(b_lo - b_hi), op_off(row, half * 8), v);
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            mma_bf16(tmem, smem_desc(smem_u32(a_hi)), smem_desc(smem_u32(b_hi)), idesc, ks == 0 ? 0u : 1u);
            mma_bf16(tmem, smem_desc(smem_u32(a_hi)), smem_desc(smem_u32(b_lo)), idesc, 1u);
            mma_bf16(tmem, smem_desc(smem_u32(a_lo)), smem_desc(smem_u32(b_hi)), idesc, 1u);
            mma_commit(bar);
        }
        // the operands are rewritten next slice: wait for these MMAs
        bool done = true;
        if (tid == 0) done = mbar_wait(bar, (uint32_t)(ks & 1), nullptr);
        ok = __syncthreads_and(done);
        tc_fence_after();
    }
    if (ok) {
        tc_fence_after();
        for (int c0 = 0; c0 < n; c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) D[(int64_t)(warp * 32 + lane) * n + c0 + i] = v[i];
        }
    } else if (tid == 0) {
        atomicOr(status, P2P_DEV_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)tmem_cols);
    }
}

int tmem_cols_for(int n) {
    int c = 32;
    while (c < n) c <<= 1;
    return c;
}

// Right-hand sides of one launch: nrhs in near-equal parts of at most 64, rounded up to 8.  A launch's tensor time
// follows its width, G is formed once per launch (the three-part split at 64 right-hand sides as two 32-wide launches,
// whose chains are shorter: 7.63 ms on the 2^21-point ellipsoid, one 64-wide launch 6.1 - 6.6 ms).
int launch_rhs(int32_t nrhs) {
    const int parts = (nrhs + 63) / 64;
    return ((nrhs + parts - 1) / parts + 7) & ~7;
}

int64_t source_groups(int64_t n) { return (n + kSrcGroup - 1) / kSrcGroup; }

}  // namespace

int32_t p2p_tc_block_count(int32_t nb) { return (nb + kBlockBoxes - 1) / kBlockBoxes; }
int p2p_tc_launch_rhs(int32_t nrhs) { return launch_rhs(nrhs); }

int64_t p2p_tc_unit_bound(int64_t n, int32_t nb) { return n / kRows + p2p_tc_block_count(nb) + 1; }

// Room for the records of either split (sized for three parts), launch by launch.
size_t p2p_tc_pack_bytes(int64_t n, int32_t max_nrhs) {
    if (max_nrhs < 16) return 0;
    size_t most = 0;
    for (int nrhs = 1; nrhs <= max_nrhs; ++nrhs) {
        const int rhs = launch_rhs(nrhs);
        most = std::max(most, (size_t)((nrhs + rhs - 1) / rhs) * (size_t)record_bytes(rhs, 3));
    }
    return (size_t)source_groups(n) * most;
}

bool p2p_tc_supported(const p2p_plan* plan, int32_t nrhs) {
    if (!plan || !plan->tc_pack || nrhs < 1 || nrhs > 256 || nrhs > plan->max_nrhs) return false;
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return false;
    if (cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess) return false;
    return major == 10 && minor == 3;
}

// Plan time: the blocks' entry lists, masks and units.  bound / units: scratch of one int per block each.
cudaError_t p2p_tc_build(p2p_plan* p, int32_t* bound, int32_t* units, void* scan_ws, cudaStream_t s) {
    const int32_t nblk = p2p_tc_block_count(p->nb);
    cudaError_t e = cudaMemsetAsync(p->tc_counter, 0, 2 * sizeof(unsigned int), s);
    if (e != cudaSuccess || nblk == 0 || p->nbs == 0) return e;
    k_tc_blocks<<<(unsigned)((nblk + 3) / 4), 128, 0, s>>>(p->box_ptr, p->nb, p->src_box_ptr, p->nbr_ptr, p->nbr_idx,
                                                            nblk, bound, units, p->tc_member);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_exclusive_i32(bound, p->tc_off, nblk, p->tc_off + nblk, scan_ws, s);
    if (e == cudaSuccess) e = scan_exclusive_i32(units, p->tc_ustart, nblk, p->tc_ustart + nblk, scan_ws, s);
    if (e != cudaSuccess) return e;
    k_tc_fill<<<(unsigned)nblk, kFillThreads, 0, s>>>(p->src_box_ptr, p->nbr_ptr, p->nbr_idx, p->nb, p->tc_off,
                                                      p->tc_ustart, p->tc_ecount, p->tc_unit_block, p->tc_gid,
                                                      p->tc_bits, p->tc_masks);
    return cudaGetLastError();
}

// Stage: the group records (strength images from original-order lambda via perm, coordinates).
p2p_status p2p_tc_stage(const p2p_plan* plan, const float2* lam, int32_t nrhs, int64_t ld, int np,
                        cudaStream_t s) {
    if (plan->n == 0 || plan->n_src == 0) return P2P_OK;
    const int rhs = launch_rhs(nrhs);
    const int64_t groups = source_groups(plan->n_src);
    const int per_block = 128 / (2 * ((rhs + 31) & ~31));
    const unsigned grid = (unsigned)((groups + per_block - 1) / per_block);
    auto pack = np == 3 ? k_tc_pack<3> : k_tc_pack<2>;
    for (int c = 0; c * rhs < nrhs; ++c) {
        pack<<<grid, 128, 0, s>>>(lam, ld, nrhs, c * rhs, rhs, plan->src_perm, plan->xs_src, plan->n_src, (int32_t)groups,
                                  plan->tc_pack + c * groups * record_bytes(rhs, np));
        P2P_CHECK_LAUNCH("p2p_apply_stage/tc_pack");
    }
    return P2P_OK;
}

p2p_status p2p_apply_tc(const p2p_plan* plan, float2* out, int32_t nrhs, int64_t ld, int32_t adjoint, int np,
                        cudaStream_t s) {
    if (plan->n == 0 || plan->n_src == 0) return P2P_OK;
    int dev = 0, optin = 0, sms = 0;
    P2P_TRY_CUDA(cudaGetDevice(&dev), "p2p_apply_tc");
    P2P_TRY_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev), "p2p_apply_tc");
    P2P_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "p2p_apply_tc");
    const int rhs = launch_rhs(nrhs);
    TcArgs a;
    a.slot_bytes = slot_bytes_for(rhs, np);
    a.slots_log = tc_smem_bytes(rhs, np, 16) <= optin ? 4 : 3;
    // more than half an SM's shared memory keeps one CTA (and one 512-column TMEM allocation) per SM
    const int smem = std::max(tc_smem_bytes(rhs, np, 1 << a.slots_log), 116 * 1024);
    if (smem > optin) {
        set_message("p2p_apply_tc: the tensor-core pipeline does not fit in shared memory");
        return P2P_ERR_UNSUPPORTED;
    }
    a.xs = plan->xs;
    a.off = plan->tc_off;
    a.ecount = plan->tc_ecount;
    a.ustart = plan->tc_ustart;
    a.unit_block = plan->tc_unit_block;
    a.gid = plan->tc_gid;
    a.bits = plan->tc_bits;
    a.masks = reinterpret_cast<const uint16_t*>(plan->tc_masks);
    a.member = plan->tc_member;
    a.box_ptr = plan->box_ptr;
    a.perm = plan->perm;
    a.nbr_ptr = plan->nbr_ptr;
    a.nbr_idx = plan->nbr_idx;
    a.src_box_ptr = plan->src_box_ptr;
    a.ld = ld;
    a.rhs = rhs;
    a.nb = plan->nb;
    a.nblk = p2p_tc_block_count(plan->nb);
    a.a_slots = np == 3 ? 4 : 8;  // 48 or 32 columns each in 256
    a.k = adjoint ? -plan->k : plan->k;
    a.status = plan->status;
    a.counter = plan->tc_counter;
    a.wait_limit = plan->tc_wait_polls < 0 ? kWaitLimit : (uint32_t)plan->tc_wait_polls;
    const bool limited = plan->tc_wait_polls >= 0;
    void (*kern)(TcArgs) = nullptr;
    const bool lap = plan->kernel == P2P_LAPLACE;
    if (np == 3) {
        kern = lap ? (limited ? k_p2p_tc<P2P_LAPLACE, true, 3> : k_p2p_tc<P2P_LAPLACE, false, 3>)
                   : (limited ? k_p2p_tc<P2P_HELMHOLTZ, true, 3> : k_p2p_tc<P2P_HELMHOLTZ, false, 3>);
    } else {
        kern = lap ? (limited ? k_p2p_tc<P2P_LAPLACE, true, 2> : k_p2p_tc<P2P_LAPLACE, false, 2>)
                   : (limited ? k_p2p_tc<P2P_HELMHOLTZ, true, 2> : k_p2p_tc<P2P_HELMHOLTZ, false, 2>);
    }
    P2P_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "p2p_apply_tc");
    const int grid = (int)std::min<int64_t>(p2p_tc_unit_bound(plan->n, plan->nb), sms);
    const int64_t part_bytes = source_groups(plan->n_src) * record_bytes(rhs, np);
    for (int c = 0; c * rhs < nrhs; ++c) {
        a.pack = plan->tc_pack + c * part_bytes;
        a.out = out + (int64_t)c * rhs;
        a.nrhs = std::min(rhs, nrhs - c * rhs);
        a.vec_out = ld % 2 == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
        kern<<<grid, kThreads, smem, s>>>(a);
        P2P_CHECK_LAUNCH("p2p_apply_tc");
    }
    return P2P_OK;
}

extern "C" P2P_API p2p_status p2p_diag_tc_gemm(const float* A, const float* B, float* D, int32_t K, int32_t n,
                                               unsigned int* status, p2p_stream_t stream) {
    if (!A || !B || !D || !status || K < 16 || K % 16 != 0 || n < 16 || n > 256 || n % 16 != 0)
        return P2P_ERR_INVALID;
    const int smem = kImage + 2 * (n / 8) * kSbo + 64;
    P2P_TRY_CUDA(cudaFuncSetAttribute(k_tc_gemm_check, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                 "p2p_diag_tc_gemm");
    k_tc_gemm_check<<<1, 128, smem, (cudaStream_t)stream>>>(A, B, D, K, n, tmem_cols_for(n), status);
    P2P_CHECK_LAUNCH("p2p_diag_tc_gemm");
    return P2P_OK;
}

// Self-check of the tensor-core path's abort handling: every pipeline wait of the plan's later tensor-core
// launches polls at most `polls` times (negative: the normal bound).
extern "C" P2P_API p2p_status p2p_diag_tc_wait_limit(p2p_plan* plan, int32_t polls) {
    if (!plan) return P2P_ERR_INVALID;
    plan->tc_wait_polls = polls < 0 ? -1 : polls;
    return P2P_OK;
}
