// SDDMM on rows that 16 bytes do not divide.  8-byte copies are compiled for
// FP32 pairs only, where they cover every even K; in 16 bits they need K to be
// a multiple of 4, and K = 100 takes 4-byte copies like the other even widths.
#include "part.cuh"
#include "sddmm_warp.cuh"

namespace spk {

cudaError_t launch_sddmm_part(int dta, int dtb, int cb, const SddmmArgs& a, cudaStream_t s)
{
    if (dta == DT_F32 && dtb == DT_F32)
        return cb == 8 ? launch_sddmm_part_cb<DT_F32, DT_F32, 8>(a, s) : launch_sddmm_part_cb<DT_F32, DT_F32, 4>(a, s);
    if (dta == DT_BF16 && dtb == DT_BF16) return launch_sddmm_part_cb<DT_BF16, DT_BF16, 4>(a, s);
    if (dta == DT_F16 && dtb == DT_F16) return launch_sddmm_part_cb<DT_F16, DT_F16, 4>(a, s);
    if (dta == DT_F32 && dtb == DT_BF16) return launch_sddmm_part_cb<DT_F32, DT_BF16, 4>(a, s);
    if (dta == DT_F32 && dtb == DT_F16) return launch_sddmm_part_cb<DT_F32, DT_F16, 4>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace spk
