// FusedMM over the balanced schedule, one warp per chunk, all heads at once
// (Sec. 2: SDDMM cascaded into SpMM on one gathered matrix B), and the first
// half of its backward, which has the same shape.
//
// The SpMM warp kernel (spmm_warp.cuh) with the scores made on the way: the
// rows of a batch of U nonzeros are copied into one of two batch slots while
// the batch before it is computed; lane l holds LB bytes of a row, so a head
// is a block of lanes.  A batch is four steps:
//   dot     a group of CL lanes holds a row, 16 bytes a lane, and makes the
//           dots of NS consecutive entries, as the SDDMM (sddmm_warp.cuh)
//           does; rows of A that start in the batch were copied with it (the
//           first NA of them).
//   reduce  NS partial dots per lane become scores: recursive halving over the
//           lanes of a head, then into shared memory.
//   weight  one lane per (head, entry): scale, value, and the row softmax as
//           a segmented maximum over the batch (segments from the mask of row
//           starts) joined with the running maximum of the row that goes on;
//           one exponential per entry and head.  The lane groups of
//           fused.cu compute it in every lane instead.
//   add     acc = acc * c + sum of w * row: the whole warp takes one row at a
//           time, LB bytes a lane, and writes a row where it ends.
// Dots in the layout of the add step (every lane 1/32 of a row) read a row
// once instead of twice but reduce every dot over 32 lanes: 16 shuffles a
// batch instead of 4 (R-MAT scale 20, BF16, K = 64, one head: 0.63 ms, this 0.52).
// Measured against the lane-group kernels of fused.cu, which stay for rows over
// 512 bytes, heads of other widths and asked-for shapes: R-MAT scale 20,
// K = 64, softmax: BF16 one head 0.94 -> 0.51 ms, FP32 4 heads with scores and
// lse 1.26 -> 0.89 ms; R-MAT of 8M nonzeros, K = 16 / 32 / 64 / 128 one head:
// FP32 0.43 / 0.54 / 0.56 / 0.95 -> 0.24 / 0.26 / 0.37 / 0.63 ms, BF16 0.70 /
// 0.49 / 0.58 / 0.75 -> 0.23 / 0.23 / 0.27 / 0.42 ms; 5 nonzeros a row, K = 64:
// 0.24 -> 0.15 and 0.28 -> 0.11 ms.  Bound by instruction issue (FP32 4 heads:
// 36 warp instructions per nonzero, issue active in half the cycles at 15 warps
// an SM, which shared memory limits).
// Backward (GRAD): A is dY, the dot is dw = <dY_i, B_j>, the weight step makes
// w (or exp(score - lse)) and c = scale * s * w * (dw - rowdot_i), writes both
// for S^T, and the add step gives dA_i = sum c B_j: one gather of B for what
// took an SDDMM, two elementwise passes and an SpMM.
#pragma once
#include "ring.cuh"
#include "sddmm_warp.cuh"
#include "spmm_warp.cuh"

namespace spk {

// The forward; the row side of the backward; the same without dA, where only
// the gradient of B is needed (4M rows with 1M entries, FP32 K = 64: the backward
// 391 us with the rows of dA stored, 213 without).
enum : int { FUSED_FORWARD = 0, FUSED_GRAD = 1, FUSED_PAIRS = 2 };

// Nonzeros per batch.  A batch costs a reduction, a weight step and the loop
// around them whatever it holds, and its slots cost resident warps; the weight
// step of one head leaves half the lanes idle at 16.  Measured (R-MAT of 8M
// nonzeros, softmax, us): forward K = 64 FP32 8 / 16 rows 487 / 376, BF16 8 / 16 /
// 32 rows 416 / 284 / 274, K = 32 16 / 32 rows FP32 302 / 255, BF16 293 / 233;
// 32 rows with 2 heads, BF16 K = 64: 316 against 277; 512-byte rows 4 / 8 rows
// 860 / 626.  Backward, 256-byte rows, 4 heads (its copies of score, lse and
// row term grow with the batch), R-MAT scale 20: 16 / 8 rows 968 / 823; the
// graph layer with 128-byte rows 16 / 32 rows 3912 / 3980 a pass.
constexpr int fused_warp_batch(bool grad, int row_bytes, int heads)
{
    if (row_bytes > (grad ? 128 : 256)) return 8;
    return !grad && heads == 1 && row_bytes <= 128 ? 32 : 16;
}

template <int DTA, int DT, int CL, int GRAD, int UB>
struct FusedWarp {
    static constexpr int RBB = CL * 16;                                       // bytes of a row of B, at most
    static constexpr int U = UB;
    static constexpr int LB = RBB / 32 > dt_bytes(DT) ? RBB / 32 : dt_bytes(DT);  // bytes of a row one lane holds
    static constexpr int E = LB / dt_bytes(DT);
    static constexpr int P = (E + 1) / 2;
    static constexpr int VA = ADot<DTA, DT>::VA;                              // vectors of A per vector of B
    static constexpr int EPI = 32 / CL, NS = U / EPI, BPT = 32 / U;
    static constexpr int SLOT = U * RBB;
    static constexpr int RA = RBB / dt_bytes(DT) * dt_bytes(DTA);             // bytes of a row of A
    static constexpr int NA = RBB >= 256 ? 4 : RBB >= 64 ? 8 : 16;            // rows of A copied with a batch
    static constexpr int VPR = RA / 16;
    static constexpr int SLOT_A = NA * RA;
    __host__ __device__ static constexpr int bytes(int heads)
    {
        // slots, weights (each twice), c and w to write out; index tiles and
        // rows of A to copy; scores, running maxima, rescale factors; scores,
        // lse and rowdot of two batches
        return 2 * (SLOT + SLOT_A) + heads * U * 8 + 4 * (2 * 32 * 3 + 2 * BPT * NA) +
               4 * heads * (GRAD ? U + 2 * U + 2 * 3 * U : U + U + 2 + 2);
    }
};

__device__ __forceinline__ int64_t fused_slot_stride(const FusedArgs& a)      // floats: K sums, (max, sum) per head
{
    return ((int64_t)a.K + 2 * a.heads + 3) / 4 * 4;
}

// One finished row of this lane's columns; lead: the first lane of a head.
template <int E>
__device__ __forceinline__ void fused_warp_row(const FusedArgs& a, bool smax, int head, bool lead, int64_t row, int col0,
                                               const float (&acc)[E], float m, float l)
{
    const bool some = !smax || l > 0.f;
    const float inv = smax && some ? 1.f / l : 1.f;
    float o[E];
#pragma unroll
    for (int q = 0; q < E; ++q) o[q] = some ? acc[q] * inv : 0.f;
    store_elems<DT_F32, E>(a.Y, row * a.ldy + col0, o);
    if (smax && a.lse && lead) a.lse[row * a.heads + head] = l > 0.f ? m + logf(l) : -INFINITY;
}

// A piece of a split row is in its carry slot: the warp that delivers the last
// one merges the pieces in slot order and writes the row.
template <int E>
__device__ __noinline__ void fused_warp_finish(const FusedArgs& a, bool smax, int head, bool lead, bool act, int col0,
                                               int s0, int64_t row)
{
    __threadfence();
    __syncwarp();
    const int lane = threadIdx.x & 31;
    int np = 0, last = 0;
    if (lane == 0) {
        np = __ldcg(a.slot_np + s0);
        last = atomicAdd(a.cnt + s0, 1) == np - 1;
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    np = __shfl_sync(0xffffffffu, np, 0);
    __threadfence();
    const int64_t sf = fused_slot_stride(a);
    if (act) {
        float M = -INFINITY, L = 0.f, sum[E];
#pragma unroll
        for (int q = 0; q < E; ++q) sum[q] = 0.f;
        const float* const ml = a.carry + a.K + 2 * head;
        if (smax)
            for (int sl = s0; sl < s0 + np; ++sl) M = fmaxf(M, __ldcg(ml + (int64_t)sl * sf));
#pragma unroll 4
        for (int sl = s0; sl < s0 + np; ++sl) {
            float c = 1.f;
            if (smax) {
                const float mp = __ldcg(ml + (int64_t)sl * sf), lp = __ldcg(ml + (int64_t)sl * sf + 1);
                c = lp > 0.f ? expf(mp - M) : 0.f;
                L += lp * c;
            }
            float x[E];
            load_elems_cg<DT_F32, E>(a.carry, (int64_t)sl * sf + col0, x);
#pragma unroll
            for (int q = 0; q < E; ++q) sum[q] = smax ? fmaf(x[q], c, sum[q]) : sum[q] + x[q];
        }
        fused_warp_row<E>(a, smax, head, lead, row, col0, sum, M, L);
    }
    __syncwarp();
    if (lane == 0) atomicExch(a.cnt + s0, 0);   // ready for the next launch
}

// FULL: a row of B is CL * 16 bytes.
template <int DTA, int DT, int CL, int GRAD, int UB, bool FULL>
__device__ __forceinline__ void fused_warp_span(const FusedArgs& a, unsigned char* wsm, const int2 b0, const int2 b1,
                                                const int4 meta, int head_s0)
{
    using W = FusedWarp<DTA, DT, CL, GRAD, UB>;
    constexpr int E = W::E, P = W::P, U = W::U, NS = W::NS, BPT = W::BPT, NA = W::NA, VA = W::VA;
    constexpr unsigned UMASK = 0xffffffffu >> (32 - U);
    const int lane = threadIdx.x & 31;
    const int e0 = b0.y, n = b1.y - b0.y;
    const int heads = a.heads;
    const bool smax = a.softmax != 0;
    const int rb = a.K * dt_bytes(DT);
    const int nhl = heads == 1 ? 32 : a.dh / E;                     // lanes of a head
    const int head = min(lane / nhl, heads - 1);
    const int col0 = lane * E;
    const bool act = (FULL && W::LB * 32 == W::RBB) || lane * W::LB < rb;
    const bool lead = act && lane == head * nhl;
    unsigned char* const slotA0 = wsm + 2 * W::SLOT;
    f32x2* const sw = reinterpret_cast<f32x2*>(slotA0 + 2 * W::SLOT_A);       // [heads][U], each twice
    int* const tcol = reinterpret_cast<int*>(sw + heads * U);       // [2][32]
    int* const trow = tcol + 64;                                    // [2][32]
    float* const tval = reinterpret_cast<float*>(trow + 64);        // [2][32]
    int* const arow = reinterpret_cast<int*>(tval + 64);            // [2][BPT][NA]: rows of A to copy
    float* const ssc = reinterpret_cast<float*>(arow + 2 * BPT * NA);         // [heads][U]
    float2* const scl = reinterpret_cast<float2*>(ssc + heads * U); // forward: [heads] factor of the row that goes on, sum of the weights
    float* const smx = reinterpret_cast<float*>(scl + heads);       // forward: [heads][1 + U] maximum before and after each entry
    float2* const scw = reinterpret_cast<float2*>(ssc + heads * U); // backward: [U][heads] c and w of the batch
    float* const sin = reinterpret_cast<float*>(scw + heads * U);                         // backward: [2][3][heads][U] score, lse, rowdot

    int nc = 0, nr = 0;
    float nv = 1.f;
    auto load_tile = [&](int i) {                                   // entry i of the chunk into this lane's registers
        if (i >= n) return;
        nc = __ldg(a.colidx + e0 + i);
        nr = __ldg(a.rowidx + e0 + i);
        if (a.vals) nv = __ldg(a.vals + e0 + i);
    };
    int last = 0;                                                   // row of the last staged entry
    auto stage = [&](int t) -> unsigned {                           // registers -> tile buffer t & 1; row-start mask
        const int o = (t & 1) * 32 + lane, i = 32 * t + lane;
        tcol[o] = nc;
        trow[o] = nr;
        tval[o] = nv;
        int up = __shfl_up_sync(0xffffffffu, nr, 1);
        if (lane == 0) up = last;
        const bool starts = i < n && nr != up;
        const unsigned m = __ballot_sync(0xffffffffu, starts);
        last = __shfl_sync(0xffffffffu, nr, 31);
        if (starts) {
            const int rank = __popc((m >> (lane / U * U)) & ((1u << (lane % U)) - 1u));
            if (rank < NA) arow[((t & 1) * BPT + lane / U) * NA + rank] = nr;
        }
        load_tile(i + 32);
        return m;
    };
    const int sub = lane / CL, vec = lane % CL;
    const bool vin = FULL || vec * 16 < rb;
    const char* __restrict__ Bb = reinterpret_cast<const char*>(a.B) + vec * 16;
    const char* __restrict__ Ab = reinterpret_cast<const char*>(a.A);
    const unsigned ldb_bytes = (unsigned)a.ldb * dt_bytes(DT);
    const unsigned lda_bytes = (unsigned)a.lda * dt_bytes(DTA);
    constexpr bool BLK = NS % 4 == 0;                               // as in the SpMM: which rows a lane copies
    const unsigned sm0 = (unsigned)__cvta_generic_to_shared(wsm);
    const unsigned slot0 = sm0 + (BLK ? sub * NS : sub) * W::RBB + vec * 16;
    const unsigned slotA = sm0 + 2 * W::SLOT + lane * 16;
    // Copy a batch: its entries are at tile-buffer offset o and from entry i of the chunk, m its row starts.
    auto issue = [&](int S, int o, int i, unsigned m) {
        const int left = n - i;
        if (left > 0) {
            const int* cols = tcol + o;
            int j[NS];
            if constexpr (BLK) {
#pragma unroll
                for (int c = 0; c < NS / 4; ++c) {
                    const int4 v = *reinterpret_cast<const int4*>(cols + sub * NS + 4 * c);
                    j[4 * c] = v.x; j[4 * c + 1] = v.y; j[4 * c + 2] = v.z; j[4 * c + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int q = 0; q < NS; ++q) j[q] = cols[q * W::EPI + sub];
            }
            constexpr int STEP = BLK ? W::RBB : W::EPI * W::RBB;
            const unsigned slot = slot0 + S * W::SLOT;
            if (FULL && left >= U) {
                for_const<NS>([&](auto q) { cpa16_at<q.value * STEP>(slot, Bb + (size_t)(unsigned)j[q.value] * ldb_bytes); });
            } else {
                for_const<NS>([&](auto q) {
                    cpa16_if<q.value * STEP>(vin && (BLK ? sub * NS + q.value : q.value * W::EPI + sub) < left, slot,
                                             Bb + (size_t)(unsigned)j[q.value] * ldb_bytes);
                });
            }
            if (m) {
                const int cnt = min(__popc(m), NA);
                const int* ar = arow + o / U * NA;
                for_const<NA * W::VPR / 32>([&](auto q) {
                    const int v = lane + 32 * q.value, r = v / W::VPR, vc = v % W::VPR;
                    const bool in = r < cnt && (FULL || vc * 16 < a.K * dt_bytes(DTA));
                    const char* p = Ab + (size_t)(unsigned)(in ? ar[r] : 0) * lda_bytes + vc * 16;
                    cpa16_if<q.value * 512>(in, slotA + S * W::SLOT_A, p);
                });
            }
            if constexpr (GRAD) {
                for (int x = lane; x < heads * U; x += 32) {
                    const int h = x / U, u = x % U;
                    if (u >= left) continue;
                    float* const d = sin + S * 3 * heads * U + x;
                    if (smax) {
                        const int64_t rh = (int64_t)trow[o + u] * heads + h;
                        cpa4(d + heads * U, a.lse + rh);
                        cpa4(d + 2 * heads * U, a.rowdot + rh);
                    }
                    cpa4(d, a.scores + (int64_t)h * a.nnz + e0 + i + u);
                }
            }
        }
        cp_async_commit();
    };

    ADot<DTA, DT> av;                                               // this lane's 16 bytes (VA x 16) of the current row of A
    const char* const Av = Ab + vec * 16 * VA;
    auto fetch_a = [&](int r) {
#pragma unroll
        for (int h = 0; h < VA; ++h) {
            ulonglong2 x = make_ulonglong2(0ull, 0ull);
            if (vin) x = __ldg(reinterpret_cast<const ulonglong2*>(Av + (size_t)(unsigned)r * lda_bytes + h * 16));
            av.set(h, x);
        }
    };
    RowAcc<DT, E> acc;
    acc.clear();
    float l = 0.f;
    int piece = meta.x >= 0;                                        // the current row goes to a carry slot
    int row = 0, slot_id = meta.x;
    auto close = [&](const float* mx) {                             // write the current row and clear it; mx: its maximum
        if (act) {
            float f[E];
            acc.get(f);
            float m = 0.f;
            if constexpr (!GRAD) m = *mx;
            if (piece) {
                float* const c = a.carry + (int64_t)slot_id * fused_slot_stride(a);
                store_elems<DT_F32, E>(c, col0, f);
                if (!GRAD && lead) {
                    c[a.K + 2 * head] = m;
                    c[a.K + 2 * head + 1] = l;
                }
            } else {
                fused_warp_row<E>(a, !GRAD && smax, head, lead, row, col0, f, m, l);
            }
        }
        piece = 0;
        l = 0.f;
        acc.clear();
    };
    const unsigned char* const read0 = wsm + lane * W::LB;
    const unsigned dotB = sm0 + sub * NS * W::RBB + vec * 16, dotA = sm0 + 2 * W::SLOT + vec * 16 * VA;
    // the lanes of a head in the dot layout, and where the reduced scores of this lane go
    const int nhv = heads == 1 ? CL : a.dh / vec_elems(DT);
    const int per = nhv >= NS ? 1 : NS / nhv;                       // entries whose scores end in one lane
    const int sidx = min(vec / nhv, heads - 1) * U + sub * NS + (nhv >= NS ? (vec % nhv) / (nhv / NS) : (vec % nhv) * per);
    const bool swr = vec < heads * nhv && (nhv < NS || (vec % nhv) % (nhv / NS) == 0);
    const f32x2* const swl = sw + head * U;
    const float* const smxl = smx + head * (U + 1);

    auto compute = [&](int S, int o, int i, unsigned m) {           // the batch at entry i of the chunk
        const int left = n - i;
        const unsigned char* const slot = read0 + S * W::SLOT;
        const unsigned slotB = dotB + S * W::SLOT, slA = dotA + S * W::SLOT_A;
        float p[NS];
        auto dots = [&](auto k) {
            typename ADot<DTA, DT>::Acc d;
            acc_zero(d);
            if (vin) av.dot(d, lds16<k.value * W::RBB>(slotB));
            p[k.value] = acc_sum(d);
        };
        auto copied = [&](int s) {
            for_const<VA>([&](auto h) { av.set(h.value, lds16<h.value * 16>(slA + s * W::RA)); });
        };
        if (m == 0) {
            for_const<NS>(dots);
        } else {
            const int cnt = __popc(m);
            const unsigned mine = m >> (sub * NS);
            int idx = __popc(m & ((1u << (sub * NS)) - 1u)) - 1;    // start that this group's first entry continues
            bool turn = idx >= 0;
            if (cnt <= NA) {
                for_const<NS>([&](auto k) {
                    if ((mine >> k.value) & 1u) { ++idx; turn = true; }
                    if (turn) copied(idx);
                    turn = false;
                    dots(k);
                });
                copied(cnt - 1);                                    // the batch's last row goes on
            } else {
                for_const<NS>([&](auto k) {
                    if ((mine >> k.value) & 1u) { ++idx; turn = true; }
                    if (turn) {
                        if (idx < NA) copied(idx);
                        else fetch_a(trow[o + sub * NS + k.value]);
                    }
                    turn = false;
                    dots(k);
                });
                fetch_a(trow[o + 31 - __clz(m)]);
            }
        }
        {
            int dd = nhv >> 1;
#pragma unroll
            for (int half = NS / 2; half >= 1; half >>= 1) {
                if (dd >= 1) {
                    const bool upper = (lane & dd) != 0;
#pragma unroll
                    for (int q = 0; q < half; ++q) {
                        const float send = upper ? p[q] : p[q + half];
                        const float keep = upper ? p[q + half] : p[q];
                        p[q] = keep + __shfl_xor_sync(0xffffffffu, send, dd);
                    }
                    dd >>= 1;
                }
            }
            for (; dd >= 1; dd >>= 1) p[0] += __shfl_xor_sync(0xffffffffu, p[0], dd);
            if (swr) {
                ssc[sidx] = p[0];
                if (per > 1) {
#pragma unroll
                    for (int q = 1; q < NS; ++q)
                        if (q < per) ssc[sidx + q] = p[q];
                }
            }
        }
        __syncwarp();
        for (int x0 = 0; x0 < heads * U; x0 += 32) {
            const int u = lane % U;
            const bool in = x0 + lane < heads * U;
            const int x = in ? x0 + lane : u;
            const int h = x / U;
            const float dotv = ssc[x], sv = tval[o + u];
            if constexpr (GRAD) {
                const float* const d = sin + S * 3 * heads * U + x;
                float w = d[0], g = dotv;
                if (smax) {
                    w = expf(w - d[heads * U]);
                    g = w * (dotv - d[2 * heads * U]);
                }
                const float c = (a.scale * sv) * g;
                if (in) {
                    sw[x] = pack2(__float_as_uint(c), __float_as_uint(c));
                    scw[u * heads + h] = make_float2(c, w);
                }
            } else {
                float s = a.scale * (sv * dotv);
                if (a.scores && in && u < left) __stcs(a.scores + (int64_t)h * a.nnz + e0 + i + u, s);
                if (smax) {
                    if (u >= left) s = -INFINITY;
                    const float mo = smx[h * (U + 1) + U];          // of the row that goes on
                    float M = s;
                    if (m == 0) {
#pragma unroll
                        for (int d = U / 2; d >= 1; d >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, d));
                        M = fmaxf(M, mo);
                    } else {
                        const unsigned upto = m & ((2u << u) - 1u), after = m & ~((2u << u) - 1u);
                        const int ss = upto ? 31 - __clz(upto) : 0;         // first entry of this entry's row
                        const int se = after ? __ffs(after) - 2 : U - 1;    // and its last one
#pragma unroll
                        for (int d = 1; d < U; d <<= 1) {
                            const float y = __shfl_up_sync(0xffffffffu, M, d, U);
                            if (u - d >= ss) M = fmaxf(M, y);
                        }
                        if (!upto) M = fmaxf(M, mo);
                        M = __shfl_sync(0xffffffffu, M, se, U);
                    }
                    s = expf(s - softmax_base(M));
                    float sum = s;
                    if (m == 0) {
#pragma unroll
                        for (int d = U / 2; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
                    }
                    __syncwarp();
                    if (in) {
                        smx[h * (U + 1) + 1 + u] = M;
                        if (u == 0) {
                            smx[h * (U + 1)] = mo;
                            scl[h] = make_float2(mo == -INFINITY ? 0.f : expf(mo - M), sum);
                        }
                    }
                }
                if (in) sw[x] = pack2(__float_as_uint(s), __float_as_uint(s));
            }
        }
        __syncwarp();
        if constexpr (GRAD) {
            float2* const out = reinterpret_cast<float2*>(a.cw) + (int64_t)(e0 + i) * heads;
            for (int x = lane; x < min(left, U) * heads; x += 32) __stcs(out + x, scw[x]);
            if constexpr (GRAD == FUSED_PAIRS) return;              // no add step
        } else if (smax && !(m & 1u)) {
            const float2 cl = scl[head];
            const f32x2 c2 = pack2(__float_as_uint(cl.x), __float_as_uint(cl.x));
            l = m == 0 && left >= U ? fmaf(l, cl.x, cl.y) : l * cl.x;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                f32x2 z = 0ull;
                ffma2(z, c2, acc.a[q]);
                acc.a[q] = z;
            }
        }
        auto four = [&](int c, bool sum) {
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                const ulonglong2 s2 = *reinterpret_cast<const ulonglong2*>(swl + c + q);
                if (!GRAD && sum) l += lo2(s2.x) + lo2(s2.y);
                acc.add(s2.x, slot + (c + q) * W::RBB);
                acc.add(s2.y, slot + (c + q + 1) * W::RBB);
            }
        };
        auto one = [&](int u) {
            if (!GRAD) l += lo2(swl[u]);
            acc.add(swl[u], slot + u * W::RBB);
        };
        auto turn_row = [&](int u) {
            close(smxl + u);
            row = trow[o + u];
        };
        if (m == 0 && left >= U) {
#pragma unroll
            for (int c = 0; c < U; c += 4) four(c, false);
        } else if (left >= U) {
#pragma unroll 1
            for (int c = 0; c < U; c += 4, m >>= 4) {
                if ((m & 15u) == 0) {
                    four(c, true);
                    continue;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((m >> q) & 1u) turn_row(c + q);
                    one(c + q);
                }
            }
        } else {
#pragma unroll 1
            for (int u = 0; u < left; ++u, m >>= 1) {
                if (m & 1u) turn_row(u);
                one(u);
            }
        }
    };
    auto zero_rows = [&]() {                                        // rows of the chunk without nonzeros
        if (GRAD == FUSED_PAIRS) return;
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
                if (act) fused_warp_row<E>(a, !GRAD && smax, head, lead, rr, col0, z, -INFINITY, 0.f);
            }
        }
    };

    if (n <= 0) {
        zero_rows();
        return;
    }
    if constexpr (!GRAD)
        for (int h = lane; h < heads; h += 32) smx[h * (U + 1) + U] = -INFINITY;
    load_tile(lane);
    last = __shfl_sync(0xffffffffu, nr, 0);                         // the first entry opens its row here
    row = last;
    unsigned mi = stage(0), mc = mi;                                // row starts of the issuing and the computing batch's tiles
    __syncwarp();
    issue(0, 0, 0, mi & UMASK);
    fetch_a(row);
    zero_rows();
    for (int i = 0, b = 0; i < n; i += U, ++b) {
        const int nx = i + U;
        if (nx % 32 == 0) {
            if (nx < n) mi = stage(nx / 32);
            __syncwarp();
        }
        issue((b & 1) ^ 1, nx % 64, nx, (mi >> (nx % 32)) & UMASK);
        cp_async_wait<1>();
        __syncwarp();
        compute(b & 1, i % 64, i, (mc >> (i % 32)) & UMASK);
        if (nx % 32 == 0) mc = mi;
        __syncwarp();                                               // the slot and the tile are read
    }
    cp_async_wait<0>();
    if (GRAD == FUSED_PAIRS) return;
    if (!piece && meta.y >= 0) {
        piece = 1;
        slot_id = meta.y;
    }
    close(smxl + U);
    if (meta.x >= 0) fused_warp_finish<E>(a, !GRAD && smax, head, lead, act, col0, head_s0, b0.x);
    if (meta.y >= 0) fused_warp_finish<E>(a, !GRAD && smax, head, lead, act, col0, meta.y, b1.x);
}

// Resident warps an SM that the registers are cut for.  More warps hide the
// latency of the gathers and of the serial steps of a batch, where shared memory
// has room for them (about 30 on rows of 64 bytes, 27 on 128 with several heads);
// with 18 in shared memory (128 bytes and one head, 256 bytes) the limit only
// changes the code.  Time over that at 20 warps (R-MAT of 4M and 8M entries, regular rows of 8 and
// 24, no spills): forward, rows of up to 64 bytes at 24 warps 0.82-0.95, at 32
// 0.80-0.92 (one head or two, FP32 and BF16); 128 bytes, FP32 at 24 0.97 one
// head, 0.82-0.88 two, at 28 1.0 / 0.82-0.9; BF16 at 24 0.98 one head, 0.82-0.94
// four, at 28 another 0.95; 256 bytes, BF16 at 24 0.92-0.97, FP32 0.99-1.01.
// Backward: up to 64 bytes at 24 0.98-1.12, at 32 0.92-1.12; BF16 rows of 128
// bytes at 28 1.03-1.06 of 24.
constexpr int fused_warp_ctas(bool grad, int dt, int cl)
{
    if (grad) return cl == 8 && dt != DT_F32 ? 24 : 20;
    if (cl <= 4) return 32;
    if (cl == 8) return dt != DT_F32 ? 28 : 24;
    return cl == 16 && dt != DT_F32 ? 24 : 20;
}

template <int DTA, int DT, int CL, int GRAD, int UB, bool FULL>
__global__ void __launch_bounds__(32, fused_warp_ctas(GRAD != FUSED_FORWARD, DT, CL))
k_fused_warp(const FusedArgs a)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const int64_t c = blockIdx.x;
    const int2 b0 = a.bnd[c], b1 = a.bnd[c + 1];
    const int4 m = a.meta[c];
    const int hs0 = (m.x >= 0) ? __ldg(a.head_s0 + c) : -1;
    fused_warp_span<DTA, DT, CL, GRAD, UB, FULL>(a, ring_smem, b0, b1, m, hs0);
}

template <int DTA, int DT, int CL, int GRAD, int UB>
cudaError_t launch_fused_warp_u(const FusedArgs& a, cudaStream_t s)
{
    using W = FusedWarp<DTA, DT, CL, GRAD, UB>;
    const bool full = a.K * dt_bytes(DT) == W::RBB;
    const void* fn = full ? (const void*)&k_fused_warp<DTA, DT, CL, GRAD, UB, true>
                          : (const void*)&k_fused_warp<DTA, DT, CL, GRAD, UB, false>;
    const size_t smem = W::bytes(a.heads);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks), dim3(32), args, smem, s);
}

template <int DTA, int DT, int CL, int GRAD>
cudaError_t launch_fused_warp_cl(const FusedArgs& a, cudaStream_t s)
{
    constexpr int U1 = fused_warp_batch(GRAD, CL * 16, 1), U2 = fused_warp_batch(GRAD, CL * 16, 2);
    return a.heads == 1 ? launch_fused_warp_u<DTA, DT, CL, GRAD, U1>(a, s) : launch_fused_warp_u<DTA, DT, CL, GRAD, U2>(a, s);
}

template <int DTA, int DT, int GRAD>
cudaError_t launch_fused_warp_dt(const FusedArgs& a, cudaStream_t s)
{
    if (a.nchunks <= 0) return cudaSuccess;
    const int rb = a.K * dt_bytes(DT);
    if (rb <= 32) return launch_fused_warp_cl<DTA, DT, 2, GRAD>(a, s);
    if (rb <= 64) return launch_fused_warp_cl<DTA, DT, 4, GRAD>(a, s);
    if (rb <= 128) return launch_fused_warp_cl<DTA, DT, 8, GRAD>(a, s);
    if (rb <= 256) return launch_fused_warp_cl<DTA, DT, 16, GRAD>(a, s);
    return launch_fused_warp_cl<DTA, DT, 32, GRAD>(a, s);
}

// Whether the warp kernels cover a call: a row of B in one block of 512 bytes,
// and heads of a power of two 16-byte vectors (one head: any width).
inline bool fused_warp_fits(int dt, int K, int heads)
{
    if (K * dt_bytes(dt) > 512) return false;
    const int dh = K / heads, nhv = dh / vec_elems(dt);
    return heads == 1 || (dh % vec_elems(dt) == 0 && (nhv & (nhv - 1)) == 0);
}

}  // namespace spk
