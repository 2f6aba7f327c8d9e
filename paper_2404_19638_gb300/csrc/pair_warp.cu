// X (+)= S_c^T A + S_w^T Y over a transpose plan: two SpMM^T that share their
// pattern and output, with the values of both as (c, w) pairs per entry and
// head in the order of S (the backward half that fused_warp.cuh leaves).
//
// One warp per chunk as in spmm_warp.cuh; a nonzero gathers a row of A and a
// row of Y (FP32) next to each other into the batch slot.  Each product has its
// own accumulator (one for both would be a chain of twice the length: 1.4 times
// the error against 64 bits), added where a row ends.  The pairs are fetched through the slot permutation where an
// index tile is staged: heads x 8 contiguous bytes an entry, so one 32-byte
// sector serves 4 heads of both products (head-major arrays: 8 sectors, and a
// permuting pass per head and product).  X is written once instead of
// written, read and written again.
#include "pair.cuh"
#include "spmm_warp.cuh"

namespace spk {

template <int DTA, int KB>
struct PairWarp {
    static constexpr int U = 512 / KB;                              // nonzeros per batch: 16, 8, 4
    static constexpr int E = KB / 32;                               // columns of a lane
    static constexpr int BPT = 32 / U;
    static constexpr int RA = KB * dt_bytes(DTA), RY = KB * 4;      // row bytes
    static constexpr int SA = U * RA, SY = U * RY, SLOT = SA + SY;
    __host__ __device__ static constexpr int bytes(int heads) { return 2 * SLOT + 2 * 32 * 4 * 2 + 2 * 32 * 8 * heads; }
};

__device__ __forceinline__ void cpa8(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

template <int E>
__device__ __noinline__ void pair_finish(const PairArgs& a, int nkb, int kbw, int s0, int64_t row)
{
    const int lane = threadIdx.x & 31;
    __threadfence();
    __syncwarp();
    int np = 0, last = 0;
    if (lane == 0) {
        np = __ldcg(a.slot_np + s0);
        last = atomicAdd(a.cnt + s0, 1) == np * nkb - 1;
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    np = __shfl_sync(0xffffffffu, np, 0);
    __threadfence();
    for (int c = lane * E; c < a.K; c += kbw) {
        float sum[E];
#pragma unroll
        for (int q = 0; q < E; ++q) sum[q] = 0.f;
#pragma unroll 4
        for (int sl = s0; sl < s0 + np; ++sl) {
            float x[E];
            load_elems_cg<DT_F32, E>(a.carry, (int64_t)sl * a.K + c, x);
#pragma unroll
            for (int q = 0; q < E; ++q) sum[q] += x[q];
        }
        if (a.accumulate) {
            float old[E];
            load_elems_cg<DT_F32, E>(a.X, row * a.ldx + c, old);
#pragma unroll
            for (int q = 0; q < E; ++q) sum[q] += old[q];
        }
        store_elems<DT_F32, E>(a.X, row * a.ldx + c, sum);
    }
    __syncwarp();
    if (lane == 0) atomicExch(a.cnt + s0, 0);   // ready for the next launch
}

// FULL: every block of KB columns is whole.
template <int DTA, int KB, bool FULL>
__global__ void __launch_bounds__(32) k_pair_warp(const PairArgs a)
{
    using W = PairWarp<DTA, KB>;
    constexpr int E = W::E, U = W::U, BPT = W::BPT;
    extern __shared__ __align__(16) unsigned char ring_smem[];
    unsigned char* const wsm = ring_smem;
    const int lane = threadIdx.x & 31;
    const int kb = blockIdx.y, nkb = gridDim.y;
    const int64_t c = blockIdx.x;
    const int2 b0 = a.bnd[c], b1 = a.bnd[c + 1];
    const int4 meta = a.meta[c];
    const int e0 = b0.y, n = b1.y - b0.y, heads = a.heads;
    const int kc = min(a.K - kb * KB, KB);                          // columns of this block
    const int col0 = kb * KB + lane * E;
    const bool act = FULL || lane * E < kc;
    int* const tcol = reinterpret_cast<int*>(wsm + 2 * W::SLOT);    // [2][32]
    int* const trow = tcol + 64;                                    // [2][32]
    float2* const tval = reinterpret_cast<float2*>(trow + 64);      // [2][32][heads]: c, w
    const int head = min(col0 / (a.K / heads), heads - 1);

    int nc = 0, nr = 0, np = 0;
    auto load_tile = [&](int i) {                                   // entry i of the chunk into this lane's registers
        if (i >= n) return;
        nc = __ldg(a.colidx + e0 + i);
        nr = __ldg(a.rowidx + e0 + i);
        np = __ldg(a.perm + e0 + i);
    };
    int last = 0;
    auto stage = [&](int t) -> unsigned {                           // tile t's pairs are copied, its rows and columns stored
        const int o = (t & 1) * 32 + lane, i = 32 * t + lane;
        tcol[o] = nc;
        trow[o] = nr;
        if (i < n) {
            const float2* src = reinterpret_cast<const float2*>(a.cw) + (int64_t)np * heads;
            for (int h = 0; h < heads; ++h) cpa8(tval + o * heads + h, src + h);
        }
        int up = __shfl_up_sync(0xffffffffu, nr, 1);
        if (lane == 0) up = last;
        const unsigned m = __ballot_sync(0xffffffffu, i < n && nr != up);
        last = __shfl_sync(0xffffffffu, nr, 31);
        load_tile(i + 32);
        return m;
    };
    constexpr int VA = W::RA / 16, VY = W::RY / 16;                 // vectors of a row
    constexpr int NA = U * VA / 32, NY = U * VY / 32;               // copies of a lane
    const char* __restrict__ Ab = reinterpret_cast<const char*>(a.A) + (int64_t)kb * W::RA + lane % VA * 16;
    const char* __restrict__ Yb = reinterpret_cast<const char*>(a.Y) + (int64_t)kb * W::RY + lane % VY * 16;
    const bool ain = FULL || lane % VA * 16 < kc * dt_bytes(DTA), yin = FULL || lane % VY * 16 < kc * 4;
    const unsigned lda_bytes = (unsigned)a.lda * dt_bytes(DTA), ldy_bytes = (unsigned)a.ldy * 4u;
    const unsigned slot0 = (unsigned)__cvta_generic_to_shared(wsm) + lane * 16;
    auto issue = [&](const int* cols, unsigned slot, int left) {
        if (left > 0) {
            if (FULL && left >= U) {
                for_const<NA>([&](auto q) {
                    cpa16_at<q.value * 512>(slot, Ab + (size_t)(unsigned)cols[lane / VA + q.value * (32 / VA)] * lda_bytes);
                });
                for_const<NY>([&](auto q) {
                    cpa16_at<W::SA + q.value * 512>(slot, Yb + (size_t)(unsigned)cols[lane / VY + q.value * (32 / VY)] * ldy_bytes);
                });
            } else {
                for_const<NA>([&](auto q) {
                    const int r = lane / VA + q.value * (32 / VA);
                    cpa16_if<q.value * 512>(ain && r < left, slot, Ab + (size_t)(unsigned)cols[r] * lda_bytes);
                });
                for_const<NY>([&](auto q) {
                    const int r = lane / VY + q.value * (32 / VY);
                    cpa16_if<W::SA + q.value * 512>(yin && r < left, slot, Yb + (size_t)(unsigned)cols[r] * ldy_bytes);
                });
            }
        }
        cp_async_commit();
    };

    RowAcc<DTA, E> accA;
    RowAcc<DT_F32, E> accY;
    accA.clear();
    accY.clear();
    float old[E];
    int piece = meta.x >= 0;
    float* dst = nullptr;
    auto open = [&](int row) {
        dst = a.X + (int64_t)row * a.ldx + col0;
        if (a.accumulate && act) load_elems_cg<DT_F32, E>(dst, 0, old);     // arrives while the row is summed
    };
    auto close = [&]() {
        if (act) {
            float f[E], g[E];
            accA.get(f);
            accY.get(g);
#pragma unroll
            for (int q = 0; q < E; ++q) f[q] += g[q];
            if (a.accumulate && !piece) {
#pragma unroll
                for (int q = 0; q < E; ++q) f[q] += old[q];
            }
            store_elems<DT_F32, E>(dst, 0, f);
        }
        piece = 0;
        accA.clear();
        accY.clear();
    };
    const unsigned char* const readA = wsm + lane * (E * dt_bytes(DTA));
    const unsigned char* const readY = wsm + W::SA + lane * (E * 4);
    auto add = [&](int S, int u, const float2* pv) {
        const float2 cw = *pv;
        accA.add(pack2(__float_as_uint(cw.x), __float_as_uint(cw.x)), readA + S * W::SLOT + u * W::RA);
        accY.add(pack2(__float_as_uint(cw.y), __float_as_uint(cw.y)), readY + S * W::SLOT + u * W::RY);
    };
    auto compute = [&](int S, int o, unsigned m, int left) {
        const float2* pv = tval + o * heads + head;
        if (m == 0 && left >= U) {
#pragma unroll
            for (int u = 0; u < U; ++u) add(S, u, pv + u * heads);
            return;
        }
        const int* rows = trow + o;
        const int cnt = min(left, U);
#pragma unroll 1
        for (int u = 0; u < cnt; ++u, m >>= 1) {
            if (m & 1u) {
                close();
                open(rows[u]);
            }
            add(S, u, pv + u * heads);
        }
    };
    auto zero_rows = [&]() {
        if (a.accumulate) return;
        float z[E];
#pragma unroll
        for (int q = 0; q < E; ++q) z[q] = 0.f;
        for (int r0 = b0.x; r0 <= meta.z; r0 += 32) {
            const int r = r0 + lane;
            bool none = false;
            if (r <= meta.z) none = __ldg(a.rowptr + r) == __ldg(a.rowptr + r + 1);
            unsigned zm = __ballot_sync(0xffffffffu, none);
            while (zm) {
                const int64_t rr = r0 + __ffs(zm) - 1;
                zm &= zm - 1;
                if (act) store_elems<DT_F32, E>(a.X, rr * a.ldx + col0, z);
            }
        }
    };
    if (n <= 0) {
        zero_rows();
        return;
    }
    auto carry_slot = [&](int slot) { return a.carry + (int64_t)slot * a.K + col0; };
    load_tile(lane);
    last = __shfl_sync(0xffffffffu, nr, 0);                         // the first entry opens its row here
    const int first = last;
    unsigned m = stage(0);
    __syncwarp();
    issue(tcol, slot0, n);
    if (piece) dst = carry_slot(meta.x);
    else open(first);
    zero_rows();
    int o = 0, left = n;
    for (int t = 0; left > 0; ++t, o ^= 32) {
        unsigned mn = 0;
#pragma unroll
        for (int q = 0; q < BPT; ++q, left -= U) {
            if (q + 1 < BPT) {
                issue(tcol + o + (q + 1) * U, slot0 + ((q + 1) & 1) * W::SLOT, left - U);
            } else {
                if (left > U) mn = stage(t + 1);
                __syncwarp();
                issue(tcol + (o ^ 32), slot0, left - U);
            }
            cp_async_wait<1>();
            __syncwarp();
            if (left > 0) compute(q & 1, o + q * U, (m >> (q * U)) & ((1u << U) - 1u), left);
            __syncwarp();                                            // the slot is read
        }
        m = mn;
    }
    cp_async_wait<0>();
    if (!piece && meta.y >= 0) {
        piece = 1;
        dst = carry_slot(meta.y);
    }
    close();
    if (meta.x >= 0) pair_finish<E>(a, nkb, KB, __ldg(a.head_s0 + c), b0.x);
    if (meta.y >= 0) pair_finish<E>(a, nkb, KB, meta.y, b1.x);
}

template <int DTA, int KB>
static cudaError_t launch_pair_kb(const PairArgs& a, cudaStream_t s)
{
    const int nkb = (a.K + KB - 1) / KB;
    if (nkb > 65535) return cudaErrorInvalidValue;
    const void* fn = a.K % KB == 0 ? (const void*)&k_pair_warp<DTA, KB, true> : (const void*)&k_pair_warp<DTA, KB, false>;
    const size_t smem = PairWarp<DTA, KB>::bytes(a.heads);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks, (unsigned)nkb), dim3(32), args, smem, s);
}

template <int DTA>
static cudaError_t launch_pair_dt(const PairArgs& a, cudaStream_t s)
{
    if (a.K <= 32) return launch_pair_kb<DTA, 32>(a, s);
    if (a.K <= 64) return launch_pair_kb<DTA, 64>(a, s);
    return launch_pair_kb<DTA, 128>(a, s);
}

cudaError_t launch_pair(int dta, const PairArgs& a, cudaStream_t s)
{
    if (a.nchunks <= 0) return cudaSuccess;
    switch (dta) {
    case DT_F32: return launch_pair_dt<DT_F32>(a, s);
    case DT_BF16: return launch_pair_dt<DT_BF16>(a, s);
    case DT_F16: return launch_pair_dt<DT_F16>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace spk
