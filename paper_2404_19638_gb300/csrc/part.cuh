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

// Where these kernels beat the element path (a lane group per chunk, lanes of
// one element, loads into registers).  A chunk belongs to a whole warp here, so
// they win by far where latency counts (small problems, 2-9 times) and while a
// gathered row takes few copies; they lose where a row takes many 8- or 4-byte
// copies, and on rows of few elements once the chip is full, where a lane group
// of 4 beats a warp.  split: some row is longer than a chunk, the sign of a
// skewed pattern, whose lane groups part at the row changes.  Time of the
// element path over that of these kernels, GB300; R-MAT with 15-16 entries a
// row, uniform rows of 23-32, bipartite of 25:
//   SpMM    FP32 K = 5: 4M entries 1.5, 1.1; 16M 1.05, 0.80, 0.85
//           FP32 K = 9-31: 1.1-2.5 at every size
//           FP32 K = 34-62, copies of 8: 4M 1.2, 1.4, 1.3; 16M 1.3, 1.3, 1.3
//           FP32 K = 47, copies of 4: 800K 1.0-1.4; 4M 0.77, 0.94, 0.84
//           FP32 K = 66, copies of 8: 100K 0.96-1.6; 4M 0.54, 1.05, 0.74
//           FP32 K = 65, copies of 4: 10K 0.85-0.9; 4M 0.34, 0.68, 0.45
//           BF16 K = 6: 4M 1.7, 1.4; 16M 1.2, 0.93, 1.0; K = 50 16M 1.9, 2.3, 2.0
//           BF16 K = 126: 4M 1.1, 1.7, 1.2; 130: 100K 0.9-1.7; 4M 0.39, 1.4, 0.49
//   SDDMM   FP32 K = 5: 4M 1.8, 1.2; 16M 0.72, 0.48, 0.53 (K = 3: 8M 1.4, 0.81)
//           FP32 K = 15 / 14: 4M 1.7, 1.4 / 2.4, 1.9; 16M 1.1, 0.85, 0.90 / 1.4, 1.1, 1.2
//           FP32 K = 29 / 30: 4M 1.3, 0.8 / 1.9, 1.4; 16M 0.74, 0.52, 0.56 / 1.0, 0.62, 0.85
//           FP32 K = 47 / 50: 16M 1.1, 1.0, 0.91 / 1.6, 1.3, 1.4
//           FP32 K = 65 / 66: 400K 1.6-2.4; 4M 0.83, 0.71, 0.71 / 1.3, 1.1, 1.2
//           FP32 K = 126, copies of 8: 4M 1.2, 0.96; 16M 0.99, 0.77, 0.90
//           BF16 K = 6: 4M 3.3, 2.5; 16M 1.2, 0.80, 0.87; wider 1.2-4 at every size
inline bool part_spmm_pays(int dt, int cb, int K, int64_t nnz, bool split)
{
    if (K <= 8) return split || nnz <= (1 << 22);
    const bool one = dt == DT_F32 && cb == 4;                 // a copy per element
    if (K <= (dt != DT_F32 ? 128 : one ? 32 : 64)) return true;
    if (one) return K <= 64 && nnz <= (1 << 20);
    return nnz <= (1 << 17);
}
// (rows of at most 512 bytes)
inline bool part_sddmm_pays(int dt, int cb, int K, int64_t nnz, bool split)
{
    const bool big = nnz > (1 << 22);
    if (dt != DT_F32) return K > 8 || split || !big;
    if (cb == 8) return !big || split || (K > 32 && K <= 80);
    if (K > 64) return nnz <= (1 << 19);
    return K > 32 || !big || (split && K <= 16 && (K > 8 || nnz <= (1 << 23)));
}

// Rows of at most 512 bytes of B (SDDMM); any K (SpMM).
cudaError_t launch_sddmm_part(int dta, int dtb, int cb, const SddmmArgs& a, cudaStream_t s);
cudaError_t launch_spmm_part(int dtb, int cb, const SpmmArgs& a, cudaStream_t s);

}  // namespace spk
