// SpMM on rows that 16 bytes do not divide (outputs of any dtype and mode).
// 8-byte copies are compiled for FP32 only (see part_sddmm.cu).
#include "part.cuh"
#include "spmm_warp.cuh"

namespace spk {

cudaError_t launch_spmm_part(int dtb, int cb, const SpmmArgs& a, cudaStream_t s)
{
    switch (dtb) {
    case DT_F32: return cb == 8 ? launch_spmm_warp<DT_F32, 8>(a, s) : launch_spmm_warp<DT_F32, 4>(a, s);
    case DT_BF16: return launch_spmm_warp<DT_BF16, 4>(a, s);
    case DT_F16: return launch_spmm_warp<DT_F16, 4>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace spk
