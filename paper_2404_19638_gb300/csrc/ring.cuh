// Ring spans for the 16-byte vector path: gathered rows travel through a
// per-warp shared-memory ring filled by cp.async, so the bytes in flight are
// bounded by shared memory instead of registers, and the index streams are
// read one tile ahead so that no gather waits on an index load.
//
// Per warp (and for each of its lane groups of G lanes, U nonzeros a batch):
//   * index tiles of RING_T = 128 nonzeros: lane l holds entries 4l..4l+3 of
//     the column (and COO row) stream as one int4 each; the tile after the
//     current one is already in registers, and a group fetches the indices of
//     its batch from the owning lane with shuffles;
//   * a ring of D batch slots.  For every nonzero of a batch, lane gl of
//     the group copies its 16-byte vectors (t*G + gl, t < NV) of the gathered
//     row into the slot and later reads back exactly those vectors, so the
//     only wait on gathered data is the lane's own cp.async.wait_group;
//   * (SDDMM) one A-row slot per group and batch: the first row that starts
//     inside the batch is copied with it; a second new row inside the same
//     batch (rare: three rows meeting within U nonzeros) is read directly;
//   * per-slot metadata (rows, values) written by the group's lanes and read
//     after a __syncwarp.
// The issue cursor runs D - 1 batches ahead of the compute cursor (D = 2 or 4
// slots per warp).
#pragma once
#include "lean.cuh"

namespace spk {

constexpr int RING_T = 128;    // nonzeros per index tile (one int4 per lane)

__device__ __forceinline__ void cpa16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cpa4(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

// Two floats in one 64-bit register pair, as the packed FMA takes them.
typedef unsigned long long f32x2;
__device__ __forceinline__ void ffma2(f32x2& acc, f32x2 s, f32x2 x)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(s), "l"(x));
}
__device__ __forceinline__ f32x2 pack2(uint32_t lo, uint32_t hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ float lo2(f32x2 x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float hi2(f32x2 x) { return __uint_as_float((uint32_t)(x >> 32)); }

// 16-byte asynchronous copy under a predicate, without a branch.
__device__ __forceinline__ void cpa16_if(bool p, unsigned smem, const void* gmem)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n @p cp.async.cg.shared.global [%0], [%1], 16;\n}\n"
                 ::"r"(smem), "l"(gmem), "r"((int)p)
                 : "memory");
}
__device__ __forceinline__ void cpa16_at(unsigned smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem), "l"(gmem) : "memory");
}

// Shared memory of one SDDMM warp with D batch slots, in bytes (host and
// device): B slots, A slots, then rows / values / second values / batch
// metadata per slot, rounded up to 128 bytes so that every warp's slots stay
// 16-byte aligned.
__host__ __device__ constexpr int sddmm_ring_bytes(int G, int NV, int U, int D)
{
    return (D * (U * NV * 512 + NV * 512 + 3 * (32 / G) * U * 4 + (32 / G) * 4) + 127) / 128 * 128;
}

// Ring kernels run 2-warp CTAs (fine occupancy steps when shared memory is
// the limit); this many fit an SM's 227 KB of shared memory, at most 16.
constexpr int RING_THREADS = 64;
__host__ __device__ constexpr int ring_min_ctas(int bytes_per_warp)
{
    return (232448 / (2 * bytes_per_warp)) > 16 ? 16
                                                 : ((232448 / (2 * bytes_per_warp)) < 1 ? 1 : (232448 / (2 * bytes_per_warp)));
}

// Tile t of a span based at tb0 (16-byte aligned): lane's four entries of
// the column and row streams; entries at or past e1 read as 0.
__device__ __forceinline__ void ring_tile(const int32_t* __restrict__ col, const int32_t* __restrict__ row, int tb0,
                                          int t, int e1, int lane, int4& c, int4& r)
{
    const int e = tb0 + t * RING_T + 4 * lane;
    if (e + 4 <= e1) {
        c = ld4(col + e);
        r = ld4(row + e);
    } else {
        c = make_int4(0, 0, 0, 0);
        r = make_int4(0, 0, 0, 0);
        if (e < e1) { c.x = __ldg(col + e); r.x = __ldg(row + e); }
        if (e + 1 < e1) { c.y = __ldg(col + e + 1); r.y = __ldg(row + e + 1); }
        if (e + 2 < e1) { c.z = __ldg(col + e + 2); r.z = __ldg(row + e + 2); }
    }
}

// Entries u = 0..U-1 of a group's batch from the tile registers of lane src0 + u/4.
template <int U>
__device__ __forceinline__ void ring_fetch(const int4& t, int src0, int (&v)[U])
{
#pragma unroll
    for (int c = 0; c < U / 4; ++c) {
        v[4 * c + 0] = __shfl_sync(0xffffffffu, t.x, src0 + c);
        v[4 * c + 1] = __shfl_sync(0xffffffffu, t.y, src0 + c);
        v[4 * c + 2] = __shfl_sync(0xffffffffu, t.z, src0 + c);
        v[4 * c + 3] = __shfl_sync(0xffffffffu, t.w, src0 + c);
    }
}

// ----------------------------------------------------------------------------
// A slice of one lane (one 16-byte vector of the row of A).  FP32 keeps the
// widened floats; BF16 / F16 keep the packed halves and multiply them with the
// packed halves of B by mixed-precision FMAs (16-bit inputs, FP32 accumulate:
// the product is exact and rounded once into the accumulator, the same result
// as an fmaf on the widened values), so neither operand is unpacked.  Both
// forms accumulate even elements in acc.x and odd ones in acc.y.
// ----------------------------------------------------------------------------
template <int DT>
struct ASlice {
    float f[4];
    __device__ __forceinline__ void set(const uint4 v)
    {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
    __device__ __forceinline__ void zero() { f[0] = f[1] = f[2] = f[3] = 0.f; }
    __device__ __forceinline__ void dot(float2& acc, const uint4 b) const
    {
        acc = __ffma2_rn(make_float2(f[0], f[1]), make_float2(__uint_as_float(b.x), __uint_as_float(b.y)), acc);
        acc = __ffma2_rn(make_float2(f[2], f[3]), make_float2(__uint_as_float(b.z), __uint_as_float(b.w)), acc);
    }
};

template <int DT>
__device__ __forceinline__ void fma_halves(float2& acc, uint32_t a, uint32_t b)
{
    if constexpr (DT == DT_BF16)
        asm("{\n .reg .b16 al, ah, bl, bh;\n mov.b32 {al, ah}, %2;\n mov.b32 {bl, bh}, %3;\n"
            " fma.rn.f32.bf16 %0, al, bl, %0;\n fma.rn.f32.bf16 %1, ah, bh, %1;\n}"
            : "+f"(acc.x), "+f"(acc.y) : "r"(a), "r"(b));
    else
        asm("{\n .reg .b16 al, ah, bl, bh;\n mov.b32 {al, ah}, %2;\n mov.b32 {bl, bh}, %3;\n"
            " fma.rn.f32.f16 %0, al, bl, %0;\n fma.rn.f32.f16 %1, ah, bh, %1;\n}"
            : "+f"(acc.x), "+f"(acc.y) : "r"(a), "r"(b));
}

template <int DT>
struct ASlice16 {
    uint4 w;
    __device__ __forceinline__ void set(const uint4 v) { w = v; }
    __device__ __forceinline__ void zero() { w = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void dot(float2& acc, const uint4 b) const
    {
        fma_halves<DT>(acc, w.x, b.x);
        fma_halves<DT>(acc, w.y, b.y);
        fma_halves<DT>(acc, w.z, b.z);
        fma_halves<DT>(acc, w.w, b.w);
    }
};
template <> struct ASlice<DT_BF16> : ASlice16<DT_BF16> {};
template <> struct ASlice<DT_F16> : ASlice16<DT_F16> {};

// ----------------------------------------------------------------------------
// SDDMM (Eq. 1) over the span [e0, e1) of one warp; DT is the dtype of both
// dense operands (F32, BF16 or F16).  ALLV: every lane's NV vectors lie
// inside K (no per-vector predicates).
//
// Rows are non-decreasing along a span, so a batch lies in one row exactly
// when its first and last nonzeros do.  Such a full batch takes the fast
// path: no per-nonzero checks, and if its row is not the row of the group's
// previous batch, that row's A slice arrives through the ring with the batch.
// Any other batch (span edge, or a row starting inside the batch) takes the
// general path: the first new row's A slice arrives through the ring, a
// second new row inside the same batch is read directly.
// ----------------------------------------------------------------------------
// NH > 0: several heads, each a block of NH consecutive 16-byte vectors of a
// row (so lane gl's vector t belongs to head (t * G + gl) / NH), one output
// array of nnz values per head (out + head * nnz); NH = 0: one dot per nonzero.
template <int DT, int G, int NV, int U, int D, bool ALLV, int NH = 0>
__device__ __forceinline__ void sddmm_ring_span(const SddmmArgs& a, int lane, unsigned char* wsm, int e0, int e1)
{
    static_assert(NH == 0 || (G % NH == 0 && (U * NV) % NH == 0), "heads must tile the lanes and the batch");
    constexpr int VECN = vec_elems(DT);
    constexpr int GPW = 32 / G;
    constexpr int WB = GPW * U;
    constexpr int BPT = RING_T / WB;
    static_assert(U % 4 == 0 && U <= G && RING_T % WB == 0, "batch shape must tile the index tile");
    if (e0 >= e1) return;
    uint4* ringB = reinterpret_cast<uint4*>(wsm);
    uint4* ringA = ringB + D * U * NV * 32;
    int* mrow = reinterpret_cast<int*>(ringA + D * NV * 32);   // [D][WB]
    float* mval = reinterpret_cast<float*>(mrow + D * WB);      // [D][WB]
    float* mval2 = mval + D * WB;                                // [D][WB]
    int* mmeta = reinterpret_cast<int*>(mval2 + D * WB);         // [D][GPW]

    const int grp = lane / G, gl = lane % G;
    const unsigned gmask = group_mask<G>(lane);
    const int nvec = a.K / VECN;
    bool vin[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t) vin[t] = ALLV || (t * G + gl) < nvec;
    const char* __restrict__ Bb = reinterpret_cast<const char*>(a.B) + gl * 16;
    const char* __restrict__ Ab = reinterpret_cast<const char*>(a.A) + gl * 16;
    const unsigned ldb_bytes = (unsigned)a.ldb * dt_bytes(DT);
    const unsigned lda_bytes = (unsigned)a.lda * dt_bytes(DT);
    const float* __restrict__ vals = a.vals;
    const float* __restrict__ vals2 = a.vals2;
    const int tb0 = e0 & ~3;
    const int nb = (e1 - tb0 + WB - 1) / WB;
    const int slot_l = grp * U + gl;                 // writer lane's metadata slot (gl < U)

    int4 tc, tr, nc, nr;
    ring_tile(a.colidx, a.rowidx, tb0, 0, e1, lane, tc, tr);
    ring_tile(a.colidx, a.rowidx, tb0, 1, e1, lane, nc, nr);
    int itile = 0;
    int ilast = -1;                       // row of this group's last scheduled nonzero

    auto issue = [&](int b) {
        if (b < nb) {
            const int t = b / BPT;
            if (t != itile) {
                tc = nc; tr = nr;
                ring_tile(a.colidx, a.rowidx, tb0, t + 1, e1, lane, nc, nr);
                itile = t;
            }
            const int src0 = ((b % BPT) * WB + grp * U) >> 2;
            int j[U], row[U];
            ring_fetch<U>(tc, src0, j);
            ring_fetch<U>(tr, src0, row);
            const int d = b % D;
            const int eg = tb0 + b * WB + grp * U;
            uint4* sB = ringB + d * U * NV * 32 + lane;
            // one decision for the whole warp: a batch that could take the
            // fast path is also right on the general one, and lock-stepped
            // groups running the two paths one after the other cost both
            const bool fast = __all_sync(0xffffffffu, (eg >= e0) && (eg + U <= e1) && (row[0] == row[U - 1]));
            if (fast) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const char* brow = Bb + (size_t)(unsigned)j[u] * ldb_bytes;
#pragma unroll
                    for (int t2 = 0; t2 < NV; ++t2)
                        if (vin[t2]) cpa16(sB + (u * NV + t2) * 32, brow + t2 * G * 16);
                }
                const bool fresh = row[0] != ilast;          // the batch starts a new row
                if (fresh) {
                    const char* arow = Ab + (size_t)(unsigned)row[0] * lda_bytes;
#pragma unroll
                    for (int t2 = 0; t2 < NV; ++t2)
                        if (vin[t2]) cpa16(ringA + (d * NV + t2) * 32 + lane, arow + t2 * G * 16);
                }
                ilast = row[0];
                if (gl < U) {
                    if (vals) cpa4(mval + d * WB + slot_l, vals + eg + gl);
                    if (vals2) cpa4(mval2 + d * WB + slot_l, vals2 + eg + gl);
                }
                if (gl == 0) mmeta[d * GPW + grp] = fresh ? 3 : 1;
            } else {
                int m = 0, prev = ilast, myrow = row[0];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (gl == u) myrow = row[u];
                    const int e = eg + u;
                    if (e < e0 || e >= e1) continue;
                    const char* brow = Bb + (size_t)(unsigned)j[u] * ldb_bytes;
#pragma unroll
                    for (int t2 = 0; t2 < NV; ++t2)
                        if (vin[t2]) cpa16(sB + (u * NV + t2) * 32, brow + t2 * G * 16);
                    m |= (row[u] != prev ? 1 : 0) << u;
                    prev = row[u];
                }
                ilast = prev;
                if (m) {
                    const int ua = __ffs(m) - 1;
                    int ra = row[0];
#pragma unroll
                    for (int u = 1; u < U; ++u)
                        if (u == ua) ra = row[u];
                    const char* arow = Ab + (size_t)(unsigned)ra * lda_bytes;
#pragma unroll
                    for (int t2 = 0; t2 < NV; ++t2)
                        if (vin[t2]) cpa16(ringA + (d * NV + t2) * 32 + lane, arow + t2 * G * 16);
                }
                if (gl < U) {
                    mrow[d * WB + slot_l] = myrow;
                    const int e = eg + gl;
                    if (e >= e0 && e < e1) {
                        if (vals) cpa4(mval + d * WB + slot_l, vals + e);
                        if (vals2) cpa4(mval2 + d * WB + slot_l, vals2 + e);
                    }
                }
                if (gl == 0) mmeta[d * GPW + grp] = m << 1;
            }
        }
        cp_async_commit();
    };

    __syncwarp();
#pragma unroll
    for (int b = 0; b < D - 1; ++b) issue(b);
    ASlice<DT> av[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t) av[t].zero();
    for (int b = 0; b < nb; ++b) {
        __syncwarp();
        issue(b + D - 1);
        cp_async_wait<D - 1>();
        __syncwarp();
        const int d = b % D;
        const int eg = tb0 + b * WB + grp * U;
        const int meta = mmeta[d * GPW + grp];
        const uint4* sB = ringB + d * U * NV * 32 + lane;
        constexpr int V = NH ? U * NV : U;               // partial dots this lane reduces
        float p[V];
        if (meta & 1) {                                  // issued on the fast path (a warp-wide decision)
            if (meta & 2) {                              // new row from nonzero 0 on: its A slice is in the ring
#pragma unroll
                for (int t = 0; t < NV; ++t)
                    if (vin[t]) av[t].set(ringA[(d * NV + t) * 32 + lane]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if constexpr (NH == 0) {
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int t = 0; t < NV; ++t)
                        if (vin[t]) av[t].dot(acc, sB[(u * NV + t) * 32]);
                    p[u] = acc.x + acc.y;
                } else {
#pragma unroll
                    for (int t = 0; t < NV; ++t) {
                        float2 acc = make_float2(0.f, 0.f);
                        if (vin[t]) av[t].dot(acc, sB[(u * NV + t) * 32]);
                        p[u * NV + t] = acc.x + acc.y;
                    }
                }
            }
        } else {
            const int m = meta >> 1;
            const int ua = m ? __ffs(m) - 1 : U;
#pragma unroll
            for (int k = 0; k < V; ++k) p[k] = 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = eg + u;
                if (e < e0 || e >= e1) continue;
                if ((m >> u) & 1) {
                    if (u == ua) {
#pragma unroll
                        for (int t = 0; t < NV; ++t)
                            if (vin[t]) av[t].set(ringA[(d * NV + t) * 32 + lane]);
                    } else {
                        const int r = mrow[d * WB + grp * U + u];
                        const uint4* arow = reinterpret_cast<const uint4*>(
                            reinterpret_cast<const char*>(a.A) + (size_t)(unsigned)r * lda_bytes) + gl;
#pragma unroll
                        for (int t = 0; t < NV; ++t)
                            if (vin[t]) av[t].set(__ldg(arow + t * G));
                    }
                }
                if constexpr (NH == 0) {
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int t = 0; t < NV; ++t)
                        if (vin[t]) av[t].dot(acc, sB[(u * NV + t) * 32]);
                    p[u] = acc.x + acc.y;
                } else {
#pragma unroll
                    for (int t = 0; t < NV; ++t) {
                        float2 acc = make_float2(0.f, 0.f);
                        if (vin[t]) av[t].dot(acc, sB[(u * NV + t) * 32]);
                        p[u * NV + t] = acc.x + acc.y;
                    }
                }
            }
        }
        if constexpr (NH > 0) {
            // Recursive halving over the NH lanes of a head block: after
            // log2(NH) levels lane gl holds C = V / NH finished dots, those of
            // values C * (gl % NH) + i, value k = u * NV + t being nonzero eg + u
            // against vector t of its row, which belongs to head
            // (t * G + gl) / NH = t * (G / NH) + gl / NH.
            constexpr int C = V / NH;
#pragma unroll
            for (int dd = NH / 2, half = V / 2; dd >= 1; dd >>= 1, half >>= 1) {
                const bool upper = (gl & dd) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const float send = upper ? p[i] : p[i + half];
                    const float keep = upper ? p[i + half] : p[i];
                    p[i] = keep + __shfl_xor_sync(gmask, send, dd, G);
                }
            }
            const int kb0 = C * (gl % NH);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int k = kb0 + i, u = k / NV, t = k % NV;
                const int ew = eg + u;
                if (ew < e0 || ew >= e1) continue;
                float sv = vals ? mval[d * WB + grp * U + u] : 1.f;
                if (vals2) sv *= mval2[d * WB + grp * U + u];
                const int head = t * (G / NH) + gl / NH;
                __stcs(a.out + (int64_t)head * a.nnz + ew, sv * p[i]);
            }
            continue;
        }
        // Reduce-scatter over the low log2(U) lane bits, then butterflies over
        // the remaining G/U lane subsets: nonzero eg + (gl % U) ends in lane gl.
#pragma unroll
        for (int dd = U / 2; dd >= 1; dd >>= 1) {
            const bool upper = (gl & dd) != 0;
#pragma unroll
            for (int i = 0; i < dd; ++i) {
                const float send = upper ? p[i] : p[i + dd];
                const float keep = upper ? p[i + dd] : p[i];
                p[i] = keep + __shfl_xor_sync(gmask, send, dd, G);
            }
        }
#pragma unroll
        for (int dd = U; dd < G; dd <<= 1) p[0] += __shfl_xor_sync(gmask, p[0], dd, G);
        const int ew = eg + gl;
        if (gl < U && ew >= e0 && ew < e1) {
            float sv = vals ? mval[d * WB + slot_l] : 1.f;
            if (vals2) sv *= mval2[d * WB + slot_l];
            __stcs(a.out + ew, sv * p[0]);
        }
    }
    cp_async_wait<0>();
}

// Shared memory of one warp of a lane-group span with two batch slots: the
// gathered rows (U rows of NV 16-byte vectors a lane), the staged COO rows and
// the staged values (two tiles of 128 entries each).
__host__ __device__ constexpr int spmm_ring_bytes(int NV, int U) { return 2 * U * NV * 32 * 16 + 4 * 128 * 4; }

}  // namespace spk
