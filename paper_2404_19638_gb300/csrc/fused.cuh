// FusedMM launches beyond the ones common.cuh declares (fused.cu).
#pragma once
#include "common.cuh"

namespace spk {

// All heads in one lane group of G lanes, NV (1 or 2) adjacent 16-byte
// vectors a lane: G * NV vectors cover a row of K, heads are blocks of
// G / heads lanes.
cudaError_t launch_fused_mh_nv(int dt, int G, int NV, const FusedArgs& a, cudaStream_t s);

// One warp per chunk, all heads (fused_warp.cu): rows of at most 512 bytes,
// heads of a power of two lanes.
bool fused_warp_supported(int dt, int K, int heads);
cudaError_t launch_fused_warp(int dt, const FusedArgs& a, cudaStream_t s);
// Its backward: a.A = dY (FP32), a.B the gathered factor of dtype dt, a.Y = dA or NULL; a.scores, a.lse and a.rowdot are read.
cudaError_t launch_fused_grad(int dt, const FusedArgs& a, cudaStream_t s);

}  // namespace spk
