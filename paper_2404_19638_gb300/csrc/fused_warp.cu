// FusedMM, one warp per chunk: forward launches (fused_warp.cuh).
#include "fused_warp.cuh"

namespace spk {

bool fused_warp_supported(int dt, int K, int heads) { return fused_warp_fits(dt, K, heads); }

cudaError_t launch_fused_warp(int dt, const FusedArgs& a, cudaStream_t s)
{
    switch (dt) {
    case DT_F32: return launch_fused_warp_dt<DT_F32, DT_F32, FUSED_FORWARD>(a, s);
    case DT_BF16: return launch_fused_warp_dt<DT_BF16, DT_BF16, FUSED_FORWARD>(a, s);
    case DT_F16: return launch_fused_warp_dt<DT_F16, DT_F16, FUSED_FORWARD>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace spk
