// Multi-head SDDMM: per head h (equal slices of K), out[h * nnz + e] =
// s_e * <A[i, head h], B[j, head h]> for every stored e = (i, j) (Eq. 1 on
// each slice), one pass over the pattern for all heads.  The warp chunk of
// the single-head SDDMM with per-head reductions (sddmm_warp.cuh, NH > 0).
#include "heads.cuh"
#include "sddmm_impl.cuh"

namespace spk {

template <int DT, int G, int NV, int U, int NH>
__global__ void __launch_bounds__(32) k_sddmm_warp_mh(const SddmmArgs a)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const int c = blockIdx.x;
    const int e0 = a.bnd[c].y, n = a.bnd[c + 1].y - e0;
    sddmm_warp_chunk<DT, DT, G, NV, U, true, NH>(a, ring_smem, e0, n);   // rows are whole lane blocks
}

// (dtype, G, NV, U, NH) compiled: the default SDDMM shapes of K = 32, 64 and
// 128 (FP32) and K = 64, 128 (BF16), every head width that tiles them.
#define SPK_SDDMM_MH(X)                                                                              \
    X(DT_F32, 8, 2, 4, 1) X(DT_F32, 8, 2, 4, 2) X(DT_F32, 8, 2, 4, 4) X(DT_F32, 8, 2, 4, 8)          \
    X(DT_F32, 4, 2, 4, 1) X(DT_F32, 4, 2, 4, 2) X(DT_F32, 4, 2, 4, 4)                                \
    X(DT_F32, 8, 4, 4, 1) X(DT_F32, 8, 4, 4, 2) X(DT_F32, 8, 4, 4, 4) X(DT_F32, 8, 4, 4, 8)          \
    X(DT_BF16, 4, 2, 4, 1) X(DT_BF16, 4, 2, 4, 2) X(DT_BF16, 4, 2, 4, 4)                             \
    X(DT_BF16, 8, 2, 4, 1) X(DT_BF16, 8, 2, 4, 2) X(DT_BF16, 8, 2, 4, 4) X(DT_BF16, 8, 2, 4, 8)

static const void* sddmm_mh_fn(int dt, int G, int NV, int U, int NH)
{
#define X(DT_, G_, NV_, U_, NH_)                                                     \
    if (dt == DT_ && G == G_ && NV == NV_ && U == U_ && NH == NH_)                   \
        return (const void*)&k_sddmm_warp_mh<DT_, G_, NV_, U_, NH_>;
    SPK_SDDMM_MH(X)
#undef X
    return nullptr;
}

bool sddmm_mh_supported(int dt, int G, int NV, int U, int NH) { return sddmm_mh_fn(dt, G, NV, U, NH) != nullptr; }

cudaError_t launch_sddmm_mh(int dt, int G, int NV, int U, int NH, const SddmmArgs& a, cudaStream_t s)
{
    const void* fn = sddmm_mh_fn(dt, G, NV, U, NH);
    if (!fn) return cudaErrorInvalidValue;
    if (a.nchunks <= 0) return cudaSuccess;
    const size_t smem = sddmm_warp_bytes(G, NV, U);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks), dim3(32), args, smem, s);
}

}  // namespace spk
