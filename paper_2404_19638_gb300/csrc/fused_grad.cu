// FusedMM backward, one warp per chunk: dA with c and w per entry and head
// (fused_warp.cuh).
#include "fused_warp.cuh"

namespace spk {

cudaError_t launch_fused_grad(int dt, const FusedArgs& a, cudaStream_t s)
{
    switch (dt) {
    case DT_F32: return a.Y ? launch_fused_warp_dt<DT_F32, DT_F32, FUSED_GRAD>(a, s) : launch_fused_warp_dt<DT_F32, DT_F32, FUSED_PAIRS>(a, s);
    case DT_BF16: return a.Y ? launch_fused_warp_dt<DT_F32, DT_BF16, FUSED_GRAD>(a, s) : launch_fused_warp_dt<DT_F32, DT_BF16, FUSED_PAIRS>(a, s);
    case DT_F16: return a.Y ? launch_fused_warp_dt<DT_F32, DT_F16, FUSED_GRAD>(a, s) : launch_fused_warp_dt<DT_F32, DT_F16, FUSED_PAIRS>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace spk
