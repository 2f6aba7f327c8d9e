// Output rows of SpMM: one finished row of C written in the output dtype,
// stored or added, and the combination of the pieces of a split row.
#pragma once
#include "common.cuh"

namespace spk {

template <int VECN>
__device__ __forceinline__ void write_vec(const SpmmArgs& a, int64_t idx, const float* v)
{
    float o[VECN];
#pragma unroll
    for (int q = 0; q < VECN; ++q) o[q] = v[q];
    switch (a.dtc) {
    case DT_BF16:
        if (a.accumulate) {
            float old[VECN];
            load_elems_cg<DT_BF16, VECN>(a.C, idx, old);
#pragma unroll
            for (int q = 0; q < VECN; ++q) o[q] += old[q];
        }
        store_elems<DT_BF16, VECN>(a.C, idx, o);
        break;
    case DT_F16:
        if (a.accumulate) {
            float old[VECN];
            load_elems_cg<DT_F16, VECN>(a.C, idx, old);
#pragma unroll
            for (int q = 0; q < VECN; ++q) o[q] += old[q];
        }
        store_elems<DT_F16, VECN>(a.C, idx, o);
        break;
    default:
        if (a.accumulate) {
            float old[VECN];
            load_elems_cg<DT_F32, VECN>(a.C, idx, old);
#pragma unroll
            for (int q = 0; q < VECN; ++q) o[q] += old[q];
        }
        store_elems<DT_F32, VECN>(a.C, idx, o);
    }
}

template <int VECN, int G, int NV>
__device__ __forceinline__ void write_row(const SpmmArgs& a, const Group<G>& g, int kb, int nvec, int64_t row,
                                          const float (&acc)[NV][VECN])
{
#pragma unroll
    for (int t = 0; t < NV; ++t) {
        const int v = kb * G * NV + t * G + g.gl;
        if (v < nvec) write_vec<VECN>(a, row * a.ldc + (int64_t)v * VECN, acc[t]);
    }
}

template <int VECN, int G, int NV>
__device__ __forceinline__ void zero_row(const SpmmArgs& a, const Group<G>& g, int kb, int nvec, int64_t row)
{
    if (a.accumulate) return;
    float z[VECN];
#pragma unroll
    for (int q = 0; q < VECN; ++q) z[q] = 0.f;
#pragma unroll
    for (int t = 0; t < NV; ++t) {
        const int v = kb * G * NV + t * G + g.gl;
        if (v < nvec) write_vec<VECN>(a, row * a.ldc + (int64_t)v * VECN, z);
    }
}

// Deposit one piece of a split row and, if it is the last to arrive, finish the row.
template <int VECN, int G, int NV>
__device__ __forceinline__ void finish_piece(const SpmmArgs& a, const Group<G>& g, int kb, int nkb, int nvec,
                                             int slot, int s0, int64_t row, const float (&acc)[NV][VECN])
{
#pragma unroll
    for (int t = 0; t < NV; ++t) {
        const int v = kb * G * NV + t * G + g.gl;
        if (v < nvec) store_elems<DT_F32, VECN>(a.carry, (int64_t)slot * a.K + (int64_t)v * VECN, acc[t]);
    }
    __threadfence();
    __syncwarp(g.mask);
    int last = 0;
    if (g.gl == 0) {
        const int np = __ldcg(a.slot_np + s0);
        const int old = atomicAdd(a.cnt + s0, 1);
        last = (old == np * nkb - 1);
    }
    last = __shfl_sync(g.mask, last, 0, G);
    if (!last) return;
    __threadfence();
    const int np = __ldcg(a.slot_np + s0);
    for (int kb2 = 0; kb2 < nkb; ++kb2) {
#pragma unroll
        for (int t = 0; t < NV; ++t) {
            const int v = kb2 * G * NV + t * G + g.gl;
            if (v >= nvec) continue;
            float sum[VECN];
#pragma unroll
            for (int q = 0; q < VECN; ++q) sum[q] = 0.f;
            for (int sl = s0; sl < s0 + np; ++sl) {
                float x[VECN];
                load_elems_cg<DT_F32, VECN>(a.carry, (int64_t)sl * a.K + (int64_t)v * VECN, x);
#pragma unroll
                for (int q = 0; q < VECN; ++q) sum[q] += x[q];
            }
            write_vec<VECN>(a, row * a.ldc + (int64_t)v * VECN, sum);
        }
    }
    __syncwarp(g.mask);
    if (g.gl == 0) atomicExch(a.cnt + s0, 0);   // ready for the next launch
}

}  // namespace spk
