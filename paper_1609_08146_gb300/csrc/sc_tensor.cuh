// sc_tensor.cuh -- device helpers of the tensor-core kernels (sc_field_tensor.cu,
// sc_idft.cu): tcgen05 wrappers (inline PTX) and the split of FP32 operands into
// two fp16 halves.  Included by those files only, after sc_field_common.cuh.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sc_field_common.cuh"

namespace sc {

namespace {

// ------------------------------------------------------------------------
// tcgen05 wrappers

// Shared-memory operand, no swizzle: core matrices of 8 x 8 halves, 128
// contiguous bytes each (MN-major: 16 bytes hold 8 M or N of one K; K-major: 8 K
// of one row); k_step bytes from one to the next along K (leading offset),
// mn_step along M or N (stride offset).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, int k_step, int mn_step)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(k_step >> 4) << 16) | ((uint64_t)(mn_step >> 4) << 32) |
           (1ull << 46);
}

// f16 x f16 -> f32, m x n, operands MN-major or K-major
__host__ __device__ constexpr uint32_t mma_idesc(int m, int n, bool a_mn, bool b_mn)
{
    return (1u << 4) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t v[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr)
                 : "memory");
}

// One look at an mbarrier's phase, without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, unsigned parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// A bounded wait of a whole warp, with the limits of mbar_wait().  That answers
// lane by lane, and in the poll where a wait runs out, or sees the abort word, one
// lane can get another answer than its neighbour; what follows a wait here are
// warp-wide instructions (tcgen05.ld, shuffles, __syncwarp), which a warp torn apart
// would never leave.  So every way out of this loop is a vote.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, unsigned parity, volatile int* s_abort, int* launch_abort,
                                          bool& timed_out)
{
    constexpr unsigned kAll = 0xffffffffu;
    const uint32_t addr = smem_u32(bar);
    uint64_t t0 = 0;
    for (unsigned it = 0; it < kSpinLimit; ++it) {
        if (__all_sync(kAll, mbar_try(addr, parity))) return true;
        if (__any_sync(kAll, *s_abort)) return false;
        if ((it & 63) == 0) {
            const uint64_t now = global_ns();
            if (it == 0) t0 = now;
            else if (__any_sync(kAll, now - t0 > kWaitNs)) break;
        }
    }
    *s_abort = 1;
    timed_out = true;
    if (launch_abort) atomicExch(launch_abort, 1);
    return false;
}

// The CTA's abort word, as one answer for the warp.
__device__ __forceinline__ bool warp_aborted(const volatile int* s_abort)
{
    return __any_sync(0xffffffffu, *s_abort != 0);
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ------------------------------------------------------------------------
// Operand splitting: eight FP32 values -> eight fp16 (16 bytes) of the high
// parts and eight of the low parts.

__device__ __forceinline__ uint32_t pack_h2(float a, float b)
{
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void split_store8(unsigned char* hi, unsigned char* lo, const float2 x[4])
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = pack_h2(x[i].x, x[i].y);
        float rx, ry;  // x - hi, exact (one mixed-precision FMA each)
        asm("{\n\t.reg .b16 a, b, m;\n\tmov.b32 {a, b}, %2;\n\tmov.b16 m, 0xBC00;\n\t"
            "fma.rn.f32.f16 %0, a, m, %3;\n\tfma.rn.f32.f16 %1, b, m, %4;\n\t}"
            : "=f"(rx), "=f"(ry)
            : "r"(h[i]), "f"(x[i].x), "f"(x[i].y));
        l[i] = pack_h2(rx, ry);
    }
    *reinterpret_cast<uint4*>(hi) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo) = make_uint4(l[0], l[1], l[2], l[3]);
}

}  // namespace

}  // namespace sc
