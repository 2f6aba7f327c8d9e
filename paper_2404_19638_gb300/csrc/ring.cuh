// Shared pieces of the kernels that stage gathered rows through shared memory
// by cp.async (spmm_warp.cuh, sddmm_warp.cuh, fused.cu), so that the bytes in
// flight are bounded by shared memory instead of registers: asynchronous
// copies, packed FP32 pairs, and the sizes of a lane-group ring.
#pragma once
#include "lean.cuh"

namespace spk {

__device__ __forceinline__ void cpa16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cpa4(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

// Two floats in one 64-bit register pair, as the packed FMA takes them.
typedef unsigned long long f32x2;
__device__ __forceinline__ void ffma2(f32x2& acc, f32x2 s, f32x2 x)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(s), "l"(x));
}
__device__ __forceinline__ f32x2 pack2(uint32_t lo, uint32_t hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ float lo2(f32x2 x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float hi2(f32x2 x) { return __uint_as_float((uint32_t)(x >> 32)); }

// 16-byte asynchronous copies with the byte offsets of both addresses in the
// instruction, unconditional or under a predicate without a branch.
template <int SO = 0, int GO = 0>
__device__ __forceinline__ void cpa16_at(unsigned smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0+%2], [%1+%3], 16;\n" ::"r"(smem), "l"(gmem), "n"(SO), "n"(GO) : "memory");
}
template <int SO = 0, int GO = 0>
__device__ __forceinline__ void cpa16_if(bool p, unsigned smem, const void* gmem)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n @p cp.async.cg.shared.global [%0+%3], [%1+%4], 16;\n}\n"
                 ::"r"(smem), "l"(gmem), "r"((int)p), "n"(SO), "n"(GO)
                 : "memory");
}

// CB (4 or 8) bytes from gmem if p, else zeros (gmem is not read).
template <int CB, int SO = 0>
__device__ __forceinline__ void cpa_part(bool p, unsigned smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0+%3], [%1], %4, %2;\n" ::"r"(smem), "l"(gmem), "r"(p ? CB : 0), "n"(SO), "n"(CB)
                 : "memory");
}

// for_const<N>(f): f(integral constant 0), ..., f(integral constant N - 1).
template <int I>
struct IntC { static constexpr int value = I; __device__ constexpr operator int() const { return I; } };
template <int N, int I = 0, typename F>
__device__ __forceinline__ void for_const(F&& f)
{
    if constexpr (I < N) {
        f(IntC<I>());
        for_const<N, I + 1>(f);
    }
}

// Ring kernels run 2-warp CTAs (fine occupancy steps when shared memory is
// the limit); this many fit an SM's 227 KB of shared memory, at most 16.
constexpr int RING_THREADS = 64;
__host__ __device__ constexpr int ring_min_ctas(int bytes_per_warp)
{
    return (232448 / (2 * bytes_per_warp)) > 16 ? 16
                                                 : ((232448 / (2 * bytes_per_warp)) < 1 ? 1 : (232448 / (2 * bytes_per_warp)));
}

// Shared memory of one warp of a lane-group span with two batch slots: the
// gathered rows (U rows of NV 16-byte vectors a lane), the staged COO rows and
// the staged values (two tiles of 128 entries each).
__host__ __device__ constexpr int spmm_ring_bytes(int NV, int U) { return 2 * U * NV * 32 * 16 + 4 * 128 * 4; }

}  // namespace spk
