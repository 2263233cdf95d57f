// What the two tensor-core kernels (p2p_tc.cu, p2p_tc_box.cu) have in common: the PTX they are made of, the operand
// layout in shared memory, and the splits into BF16 parts.
#pragma once

#include <cuda_bf16.h>

#include "p2p_internal.cuh"

namespace p2p_tc_common {

constexpr float kInv4Pi = 0.0795774715459476679f;
constexpr int kSrcGroup = 16;          // sources per stage (MMA K)
constexpr int kPart = 4096;            // one BF16 image of a 128 x 16 A operand
constexpr int kLbo = 128, kSbo = 256;  // core-matrix strides (K direction, 8-row groups)
// A waiting thread is suspended (up to kSuspendNs per poll) until the phase
// completes, so idle roles do not take issue slots from the working warps.
// kWaitLimit polls bound every wait to a few seconds at most.
constexpr uint32_t kSuspendNs = 10000;
constexpr uint32_t kWaitLimit = 1u << 18;
constexpr uint32_t kDrainLimit = 1u << 14;

// --------------------------------------------------------------- PTX helpers --

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start, leading and stride byte offsets (>> 4),
// descriptor version 1 at bit 46, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kLbo >> 4) << 16) | ((uint64_t)(kSbo >> 4) << 32) |
           (1ull << 46);
}

// Instruction descriptor of kind::f16: D f32, A and B bf16, both K-major, N, M = 128.
__host__ __device__ inline uint32_t idesc_bf16_f32(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The two BF16 values of a word, as floats.
__device__ __forceinline__ float2 unpack_bf16(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ uint32_t pack_bf16(float2 v) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// v - w, exactly where w is v's rounding (one packed operation).
__device__ __forceinline__ float2 residual(float2 v, float2 w) { return __ffma2_rn(w, make_float2(-1.f, -1.f), v); }

// The largest finite BF16 value.  A finite strength above it (up to 0.4 % below the FP32 maximum) would round to infinity,
// and 0 x inf reaches targets that are not its neighbours; capped, the next part holds the rest of it.
constexpr float kBf16Max = 3.3895313892515355e38f;
__device__ __forceinline__ float capped(float x) { return isfinite(x) ? fminf(fmaxf(x, -kBf16Max), kBf16Max) : x; }

// Whether some of eight values would round to infinity in BF16 (or is infinite); splitting them takes the capped form then.
__device__ __forceinline__ bool any_above(const float (&v)[8]) {
    float m = fabsf(v[0]);
#pragma unroll
    for (int i = 1; i < 8; ++i) m = fmaxf(m, fabsf(v[i]));
    return m > kBf16Max;
}

// x = hi + lo with hi, lo BF16 (round to nearest), two values per 32-bit word.  CAP: any finite x.
template <bool CAP = false>
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    const float2 v = make_float2(a, b);
    hi = pack_bf16(CAP ? make_float2(capped(a), capped(b)) : v);
    lo = pack_bf16(residual(v, unpack_bf16(hi)));
}

// x = hi + mid + lo with three BF16 parts (each the round-to-nearest of what the
// previous parts leave), two values per 32-bit word: the parts carry ~24 bits.
template <bool CAP = false>
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    const float2 v = make_float2(a, b);
    hi = pack_bf16(CAP ? make_float2(capped(a), capped(b)) : v);
    const float2 r = residual(v, unpack_bf16(hi));
    mid = pack_bf16(r);
    lo = pack_bf16(residual(r, unpack_bf16(mid)));
}

// Byte offset of element (row, k) of a K-major operand with 16-wide K slices.
__host__ __device__ inline int op_off(int row, int k) {
    return (row >> 3) * kSbo + (k >> 3) * kLbo + (row & 7) * 16 + (k & 7) * 2;
}

}  // namespace p2p_tc_common
