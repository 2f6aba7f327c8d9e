// Paired S^T products (pair_warp.cu).
#pragma once
#include "common.cuh"

namespace spk {

struct PairArgs {
    int32_t K, heads, accumulate;
    const int32_t* rowptr;                // of S^T
    const int32_t* colidx;
    const int32_t* rowidx;
    const int32_t* perm;                  // entry of S each entry of S^T is
    const float* cw;                      // nnz x heads pairs (c, w), in S's entry order
    const void* A; int64_t lda;           // rows multiplied by c
    const float* Y; int64_t ldy;          // rows multiplied by w
    float* X; int64_t ldx;
    const int2* bnd;
    const int4* meta;
    const int32_t* head_s0;
    const int32_t* slot_np;
    int32_t* cnt;
    float* carry;                         // K floats per slot
    int64_t nchunks;
};
cudaError_t launch_pair(int dta, const PairArgs& a, cudaStream_t s);

}  // namespace spk
