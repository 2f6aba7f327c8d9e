// SDDMM and SpMM on rows that 16 bytes do not divide (part_*.cu): the warp
// kernels with copies of 4 or 8 bytes.
#pragma once
#include "common.cuh"

namespace spk {

// Bytes of a copy that rows of K elements at p with stride ld allow: 8 or 4,
// or 0 where rows start at odd 2-byte (or 1-byte) offsets, and for E4M3.
inline int part_bytes(int dt, const void* p, int64_t ld, int K)
{
    if (dt == DT_E4M3) return 0;
    const int64_t all = (int64_t)(reinterpret_cast<uintptr_t>(p) | (uintptr_t)(ld * dt_bytes(dt)) | (uintptr_t)(K * dt_bytes(dt)));
    return all % 8 == 0 ? 8 : (all % 4 == 0 ? 4 : 0);
}

// Rows of at most 512 bytes of B (SDDMM); any K (SpMM).
cudaError_t launch_sddmm_part(int dta, int dtb, int cb, const SddmmArgs& a, cudaStream_t s);
cudaError_t launch_spmm_part(int dtb, int cb, const SpmmArgs& a, cudaStream_t s);

}  // namespace spk
