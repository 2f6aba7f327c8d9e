// SDDMM over the balanced schedule, one warp per chunk (Sec. 3.2, Eq. 1).
//
// A warp batch is 32/G lane groups of U consecutive nonzeros; lane gl of a
// group holds the 16-byte vectors t * G + gl (t < NV) of a row.  Every lane
// copies the vectors of B that it reads back itself by cp.async, one batch
// ahead, into one of two batch slots.
//
// Rows of A: the entries that start a row are known per 32-entry index tile
// from one ballot, so the rows that start inside a batch are copied with the
// batch, one per lane group (32/G of them, a row for every U entries).  A
// batch without a row start multiplies with the A slice in registers.  In any
// other batch every group counts the row starts up to its entries and takes
// its slices from those copies by predicated shared loads; only rows beyond
// the 32/G copied ones (rows of fewer than U entries) are read from global
// memory.  Groups that pick rows by comparing row ids entry by entry run one
// after another: that took two thirds of the instructions on R-MAT scale 20.
//
// Outputs are per nonzero, so chunks and groups never combine results.  The
// order of each dot (even and odd elements apart, vectors in order, then the
// reduce-scatter over the lanes) is that of the register path, bit for bit.
//
// Rows that 16 bytes do not divide (CB < 16): a lane copies its vectors 8 or 4
// bytes at a time, zeros past the end of a row; the dots are the same.
// The element path, 4 bytes a lane into registers: 210 us against 129 (120,011 x
// 75,503, 20 nonzeros a row, FP32, K = 50).
//
// What bounds it (GB300): FP32 rows the shared-memory data path (64-78 %
// busy) and the latency of the gathers at the 18 warps an SM has room for;
// 16-bit rows that latency and the issue of one mixed-precision FMA per
// element.  Measured on R-MAT scale 20, K = 64, lane groups comparing rows
// entry by entry / this: FP32 0.359 / 0.298 ms (239 / 141 M instructions),
// BF16 0.228 / 0.212 ms (107 M); FP32 x BF16 0.257 ms; E4M3 K = 128 0.334 ms.
// Other shapes: FP32 16 lanes x 1 vector 0.318 ms, BF16 8 x 1 0.218 ms.  L2
// prefetch of the index streams 64-256 entries ahead: no gain.  Shared
// addresses and offsets are in the instructions (cpa16_at, lds16): the same
// loop with computed addresses took 0.324 ms.
#pragma once
#include "ring.cuh"

namespace spk {

// One lane's slice of a row of A against one 16-byte vector of B, even
// elements into acc.x and odd ones into acc.y, each product rounded once into
// its FP32 accumulator.  VA: 16-byte vectors of A per vector of B.
template <int DTA, int DTB>
struct ADot;

// 16 bytes as two 64-bit register pairs, the operands of the packed FMA.
template <int OFF = 0>
__device__ __forceinline__ ulonglong2 lds16(unsigned smem)
{
    ulonglong2 v;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(v.x), "=l"(v.y) : "r"(smem), "n"(OFF) : "memory");
    return v;
}
__device__ __forceinline__ uint4 words(const ulonglong2 v)
{
    return make_uint4((uint32_t)v.x, (uint32_t)(v.x >> 32), (uint32_t)v.y, (uint32_t)(v.y >> 32));
}

// The first n of 16 bytes at p, CB bytes a load, zeros after them.
template <int CB>
__device__ __forceinline__ ulonglong2 ldg_part(const char* p, int n)
{
    uint32_t w[4];
#pragma unroll
    for (int c = 0; c < 16; c += 4) w[c / 4] = c / CB * CB < n ? __ldg(reinterpret_cast<const unsigned int*>(p + c)) : 0u;
    return make_ulonglong2(pack2(w[0], w[1]), pack2(w[2], w[3]));
}

template <>
struct ADot<DT_F32, DT_F32> {
    static constexpr int VA = 1;
    using Acc = f32x2;
    ulonglong2 v;
    __device__ __forceinline__ void set(int, const ulonglong2 x) { v = x; }
    __device__ __forceinline__ void dot(f32x2& acc, const ulonglong2 b) const
    {
        ffma2(acc, v.x, b.x);
        ffma2(acc, v.y, b.y);
    }
};

// 16-bit operands stay packed: mixed-precision FMAs (16-bit inputs, FP32
// accumulate) round like an fmaf on the widened values.
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
struct ADot16 {
    static constexpr int VA = 1;
    using Acc = float2;
    uint4 w;
    __device__ __forceinline__ void set(int, const ulonglong2 v) { w = words(v); }
    __device__ __forceinline__ void dot(float2& acc, const ulonglong2 v) const
    {
        const uint4 b = words(v);
        fma_halves<DT>(acc, w.x, b.x);
        fma_halves<DT>(acc, w.y, b.y);
        fma_halves<DT>(acc, w.z, b.z);
        fma_halves<DT>(acc, w.w, b.w);
    }
};
template <> struct ADot<DT_BF16, DT_BF16> : ADot16<DT_BF16> {};
template <> struct ADot<DT_F16, DT_F16> : ADot16<DT_F16> {};

// FP32 rows of A against 16-bit rows of B.
template <int DTB>
struct ADotMixed {
    static constexpr int VA = 2;
    using Acc = f32x2;
    f32x2 a[4];
    __device__ __forceinline__ void set(int h, const ulonglong2 x)
    {
        a[2 * h] = x.x;
        a[2 * h + 1] = x.y;
    }
    __device__ __forceinline__ void dot(f32x2& acc, const ulonglong2 v) const
    {
        const uint4 b = words(v);
        Raw<DTB, 8> r;
        r.w[0] = b.x; r.w[1] = b.y; r.w[2] = b.z; r.w[3] = b.w;
        float f[8];
        unpack_all<DTB, 8>(r, f);
#pragma unroll
        for (int q = 0; q < 4; ++q) ffma2(acc, a[q], pack2(__float_as_uint(f[2 * q]), __float_as_uint(f[2 * q + 1])));
    }
};
template <> struct ADot<DT_F32, DT_BF16> : ADotMixed<DT_BF16> {};
template <> struct ADot<DT_F32, DT_F16> : ADotMixed<DT_F16> {};

// E4M3 codes are FP16 values: widened in pairs, then the FP16 products above.
template <>
struct ADot<DT_E4M3, DT_E4M3> {
    static constexpr int VA = 1;
    using Acc = float2;
    uint32_t h[8];
    __device__ __forceinline__ void set(int, const ulonglong2 x)
    {
        const uint4 v = words(x);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) e4m3x4_to_f16x2(w[q], h[2 * q], h[2 * q + 1]);
    }
    __device__ __forceinline__ void dot(float2& acc, const ulonglong2 v) const
    {
        const uint4 b = words(v);
        const uint32_t w[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t lo, hi;
            e4m3x4_to_f16x2(w[q], lo, hi);
            fma_halves<DT_F16>(acc, h[2 * q], lo);
            fma_halves<DT_F16>(acc, h[2 * q + 1], hi);
        }
    }
};

__device__ __forceinline__ void acc_zero(f32x2& a) { a = 0ull; }
__device__ __forceinline__ void acc_zero(float2& a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ float acc_sum(const f32x2& a) { return lo2(a) + hi2(a); }
__device__ __forceinline__ float acc_sum(const float2& a) { return a.x + a.y; }

template <int DTA, int DTB, int G, int NV, int U>
struct SddmmWarp {
    static constexpr int GPW = 32 / G;                   // lane groups; also the A rows copied with a batch
    static constexpr int WB = GPW * U;                   // nonzeros of a warp batch
    static constexpr int BPT = 32 / WB;                  // batches per index tile
    static constexpr int VA = ADot<DTA, DTB>::VA;
    static constexpr int SLOT_B = U * NV * 512, SLOT_A = NV * VA * 512;
    static constexpr int SCALES = DTB == DT_E4M3 ? 1 : 0;
    static_assert(U % 4 == 0 && U <= G && WB <= 32, "batches must tile the index tile; U lanes store results");
    // two batch slots; two tiles of columns, rows, values (and scales), and the A rows of their batches
    static constexpr int BYTES = 2 * (SLOT_B + SLOT_A) + 2 * 4 * (32 * (3 + SCALES) + 32 / U);
};
__host__ __device__ constexpr int sddmm_warp_bytes(int G, int NV, int U)      // A and B of one dtype, no scales
{
    return 2 * (U * NV * 512 + NV * 512) + 2 * 4 * (32 * 3 + 32 / U);
}

// The chunk's nonzeros [e0, e0 + n).  ALLV: every lane's NV vectors lie inside
// K.  NH > 0: several heads, each a block of NH consecutive vectors of a row
// (lane gl's vector t belongs to head (t * G + gl) / NH), one output array of
// nnz values per head; NH = 0: one dot per nonzero.  CB: bytes of a copy
// (below 16, ALLV is false).
template <int DTA, int DTB, int G, int NV, int U, bool ALLV, int NH = 0, int CB = 16>
__device__ __forceinline__ void sddmm_warp_chunk(const SddmmArgs& a, unsigned char* wsm, int e0, int n)
{
    using W = SddmmWarp<DTA, DTB, G, NV, U>;
    static_assert(NH == 0 || (G % NH == 0 && (U * NV) % NH == 0), "heads must tile the lanes and the batch");
    constexpr int GPW = W::GPW, WB = W::WB, BPT = W::BPT, VA = W::VA, NA = GPW;
    constexpr unsigned WMASK = WB == 32 ? 0xffffffffu : (1u << (WB % 32)) - 1u;
    if (n <= 0) return;
    const int lane = threadIdx.x & 31, grp = lane / G, gl = lane % G;
    const int nvec = (a.K + vec_elems(DTB) - 1) / vec_elems(DTB);
    const int rowA = a.K * dt_bytes(DTA), rowB = a.K * dt_bytes(DTB);
    bool vin[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t) vin[t] = ALLV || t * G + gl < nvec;
    unsigned char* const slotA0 = wsm + 2 * W::SLOT_B;
    int* const tcol = reinterpret_cast<int*>(slotA0 + 2 * W::SLOT_A);      // [2][32]
    int* const trow = tcol + 64;                                           // [2][32]
    float* const tval = reinterpret_cast<float*>(trow + 64);               // [2][32]
    float* const tscl = tval + 64;                                         // [2][32], E4M3 only
    int* const arow = reinterpret_cast<int*>(tval + 64 + 64 * W::SCALES);  // [2][BPT][NA]: A rows to copy
    const char* __restrict__ Bb = reinterpret_cast<const char*>(a.B) + gl * 16;
    const char* __restrict__ Ab = reinterpret_cast<const char*>(a.A) + gl * 16 * VA;
    const unsigned ldb_bytes = (unsigned)a.ldb * dt_bytes(DTB);
    const unsigned lda_bytes = (unsigned)a.lda * dt_bytes(DTA);
    const unsigned smB = (unsigned)__cvta_generic_to_shared(wsm) + lane * 16;
    const unsigned smA = smB + 2 * W::SLOT_B, smA0 = smA - grp * G * 16;      // copy: this group's; copy 0

    int nc = 0, nr = 0;
    float nv = 1.f, ns = 1.f;
    auto load_tile = [&](int i) {                        // entry i of the chunk into this lane's registers
        if (i >= n) return;
        const int e = e0 + i;
        nc = __ldg(a.colidx + e);
        nr = __ldg(a.rowidx + e);
        if (a.vals) nv = __ldg(a.vals + e);
        if (a.vals2) nv = (a.vals ? nv : 1.f) * __ldg(a.vals2 + e);
        if constexpr (DTB == DT_E4M3) ns = __ldg(a.a_scale + nr) * __ldg(a.b_scale + nc);
    };
    int last = -1;                                       // row of the last staged entry (none: the first starts a row)
    auto stage = [&](int t) -> unsigned {                // registers -> tile buffer t & 1; row-start mask
        const int o = (t & 1) * 32 + lane, i = 32 * t + lane;
        tcol[o] = nc;
        trow[o] = nr;
        tval[o] = nv;
        if constexpr (DTB == DT_E4M3) tscl[o] = ns;
        int up = __shfl_up_sync(0xffffffffu, nr, 1);
        if (lane == 0) up = last;
        const bool starts = i < n && nr != up;
        const unsigned m = __ballot_sync(0xffffffffu, starts);
        last = __shfl_sync(0xffffffffu, nr, 31);
        if (starts) {
            // the first NA - 1 rows that start in a batch, and the last one, have a copy
            const int b = lane / WB;
            const unsigned mb = (m >> (b * WB)) & WMASK;
            const int rank = __popc(mb & ((1u << (lane % WB)) - 1u)), cnt = __popc(mb);
            int* ar = arow + ((t & 1) * BPT + b) * NA;
            if (rank < NA - 1) ar[rank] = nr;
            else if (rank == cnt - 1) ar[NA - 1] = nr;
        }
        load_tile(i + 32);
        return m;
    };
    // Copy the rows of the batch at tile-buffer offset o, `left` (or WB) entries
    // of which exist, into slot S.
    auto issue = [&](auto S, int o, int left, unsigned mb) {
        constexpr int SB = S.value * W::SLOT_B, SA = S.value * W::SLOT_A;
        if (left > 0) {
            int j[U];
#pragma unroll
            for (int c = 0; c < U / 4; ++c) {
                const int4 v = *reinterpret_cast<const int4*>(tcol + o + grp * U + 4 * c);
                j[4 * c] = v.x; j[4 * c + 1] = v.y; j[4 * c + 2] = v.z; j[4 * c + 3] = v.w;
            }
            const bool whole = ALLV && left >= WB;
            if constexpr (CB < 16) {
                for_const<U>([&](auto u) {
                    const bool on = grp * U + u.value < left;
                    const char* p = Bb + (on ? (size_t)(unsigned)j[u.value] * ldb_bytes : 0);
                    for_const<NV * (16 / CB)>([&](auto q) {
                        constexpr int t = q.value / (16 / CB), o = t * G * 16 + q.value % (16 / CB) * CB;
                        const bool in = on && gl * 16 + o < rowB;
                        cpa_part<CB, SB + (u.value * NV + t) * 512 + q.value % (16 / CB) * CB>(in, smB, in ? p + o : Bb);
                    });
                });
            } else if (whole) {
                for_const<U>([&](auto u) {
                    const char* p = Bb + (size_t)(unsigned)j[u.value] * ldb_bytes;
                    for_const<NV>([&](auto t) {
                        cpa16_at<SB + (u.value * NV + t.value) * 512, t.value * G * 16>(smB, p);
                    });
                });
            } else {
                for_const<U>([&](auto u) {
                    const char* p = Bb + (size_t)(unsigned)j[u.value] * ldb_bytes;
                    for_const<NV>([&](auto t) {
                        cpa16_if<SB + (u.value * NV + t.value) * 512, t.value * G * 16>(
                            vin[t.value] && grp * U + u.value < left, smB, p);
                    });
                });
            }
            if (mb) {
                const int cnt = __popc(mb);
                // group g copies start g; the last group the last start, if it is not among the first NA - 1
                const bool mine = grp < NA - 1 ? grp < cnt : cnt >= NA;
                const int r = mine ? arow[o / WB * NA + grp] : 0;
                const char* p = Ab + (size_t)(unsigned)r * lda_bytes;
                if constexpr (CB < 16)
                    for_const<NV * VA * (16 / CB)>([&](auto q) {
                        constexpr int v = q.value / (16 / CB), c = q.value % (16 / CB) * CB;
                        constexpr int o = v / VA * G * 16 * VA + v % VA * 16 + c;
                        const bool in = mine && gl * 16 * VA + o < rowA;
                        cpa_part<CB, SA + v * 512 + c>(in, smA, in ? p + o : Ab);
                    });
                else
                for_const<NV * VA>([&](auto q) {
                    constexpr int t = q.value / VA, h = q.value % VA;
                    cpa16_if<SA + q.value * 512, t * G * 16 * VA + h * 16>(mine && vin[t], smA, p);
                });
            }
        }
        cp_async_commit();
    };

    ADot<DTA, DTB> av[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t)
#pragma unroll
        for (int h = 0; h < VA; ++h) av[t].set(h, make_ulonglong2(0ull, 0ull));
    float* const outg = a.out + e0 + grp * U;            // where this group's first entry of a batch goes
    auto compute = [&](auto S, int o, int b0, int left, unsigned mb) {   // the batch starts at entry b0 of the chunk
        constexpr int SB = S.value * W::SLOT_B, SA = S.value * W::SLOT_A;
        constexpr int V = NH ? U * NV : U;               // partial dots this lane reduces
        float p[V];
        auto dots = [&](auto u) {
            typename ADot<DTA, DTB>::Acc acc;
            acc_zero(acc);
            for_const<NV>([&](auto t) {
                if (vin[t.value]) av[t.value].dot(acc, lds16<SB + (u.value * NV + t.value) * 512>(smB));
                if constexpr (NH > 0) {
                    p[u.value * NV + t.value] = acc_sum(acc);
                    acc_zero(acc);
                }
            });
            if constexpr (NH == 0) p[u.value] = acc_sum(acc);
        };
        auto copied = [&](int s) {                       // A slice from copy s of this batch
            for_const<NV * VA>([&](auto q) { av[q.value / VA].set(q.value % VA, lds16<SA + q.value * 512>(smA0 + s * G * 16)); });
        };
        if (mb == 0) {
            for_const<U>(dots);
        } else {
            const int cnt = __popc(mb);
            const unsigned mine = mb >> (grp * U);
            int idx = __popc(mb & ((1u << (grp * U)) - 1u)) - 1;       // start that this group's first entry continues
            bool turn = idx >= 0;
            if (cnt <= NA) {
                for_const<U>([&](auto u) {
                    if ((mine >> u.value) & 1u) { ++idx; turn = true; }
                    if (turn) copied(idx);
                    turn = false;
                    dots(u);
                });
            } else {                                     // rows of fewer than U entries on average
                for_const<U>([&](auto u) {
                    if ((mine >> u.value) & 1u) { ++idx; turn = true; }
                    if (turn) {
                        if (idx < NA - 1 || idx == cnt - 1) {
                            copied(min(idx, NA - 1));
                        } else {
                            const char* q = Ab + (size_t)(unsigned)trow[o + grp * U + u.value] * lda_bytes;
#pragma unroll
                            for (int t = 0; t < NV; ++t)
                                if (vin[t])
#pragma unroll
                                    for (int h = 0; h < VA; ++h) {
                                        const char* x = q + t * G * 16 * VA + h * 16;
                                        if constexpr (CB < 16) av[t].set(h, ldg_part<CB>(x, rowA - (gl * 16 * VA + t * G * 16 * VA + h * 16)));
                                        else av[t].set(h, __ldg(reinterpret_cast<const ulonglong2*>(x)));
                                    }
                        }
                    }
                    turn = false;
                    dots(u);
                });
            }
            copied(min(cnt, NA) - 1);                    // the batch's last row goes on
        }
        const float* const sv = tval + o + grp * U;
        const int mine_left = left - grp * U;            // entries of this group
        if constexpr (NH > 0) {
            // Recursive halving over the NH lanes of a head block: after
            // log2(NH) levels lane gl holds C = V / NH finished dots, those of
            // values C * (gl % NH) + i, value k = u * NV + t being entry u
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
                    p[i] = keep + __shfl_xor_sync(0xffffffffu, send, dd);
                }
            }
            const int kb0 = C * (gl % NH);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int k = kb0 + i, u = k / NV, t = k % NV;
                if (u >= mine_left) continue;
                const int head = t * (G / NH) + gl / NH;
                __stcs(outg + (int64_t)head * a.nnz + b0 + u, sv[u] * p[i]);
            }
            return;
        }
        // Reduce-scatter over the low log2(U) lane bits, then butterflies over
        // the remaining G/U lane subsets: entry gl % U ends in lane gl.
#pragma unroll
        for (int dd = U / 2; dd >= 1; dd >>= 1) {
            const bool upper = (gl & dd) != 0;
#pragma unroll
            for (int i = 0; i < dd; ++i) {
                const float send = upper ? p[i] : p[i + dd];
                const float keep = upper ? p[i + dd] : p[i];
                p[i] = keep + __shfl_xor_sync(0xffffffffu, send, dd);
            }
        }
#pragma unroll
        for (int dd = U; dd < G; dd <<= 1) p[0] += __shfl_xor_sync(0xffffffffu, p[0], dd);
        if (gl < U && gl < mine_left) {
            float r = p[0];
            if constexpr (DTB == DT_E4M3) r *= tscl[o + grp * U + gl];
            __stcs(outg + b0 + gl, sv[gl] * r);
        }
    };

    load_tile(lane);
    unsigned mi = stage(0), mc = mi;                     // row starts of the issuing and the computing batch's tiles
    __syncwarp();
    issue(IntC<0>(), 0, n, mi & WMASK);
    for (int b0 = 0; b0 < n; b0 += 2 * WB) {
        for_const<2>([&](auto S) {
            const int b = b0 + S.value * WB;             // this batch and the next, as entries of the chunk
            const int nx = b + WB;
            const unsigned mb = (mc >> (b % 32)) & WMASK;
            if (nx % 32 == 0) {
                if (nx < n) mi = stage(nx / 32);
                __syncwarp();
            }
            issue(IntC<1 - S.value>(), nx % 64, n - nx, (mi >> (nx % 32)) & WMASK);
            cp_async_wait<1>();
            __syncwarp();
            if (b < n) compute(S, b % 64, b, n - b, mb);
            if (nx % 32 == 0) mc = mi;
            __syncwarp();                                // the slot and the tile are read
        });
    }
    cp_async_wait<0>();
}

// One warp per CTA and chunk, so that every per-chunk quantity is uniform.
template <int DTA, int DTB, int G, int NV, int U, int CB>
__global__ void __launch_bounds__(32) k_sddmm_warp_part(const SddmmArgs a)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const int e0 = a.bnd[blockIdx.x].y;
    sddmm_warp_chunk<DTA, DTB, G, NV, U, false, 0, CB>(a, ring_smem, e0, a.bnd[blockIdx.x + 1].y - e0);
}

template <int DTA, int DTB, int G, int NV, int U>
__global__ void __launch_bounds__(32) k_sddmm_warp(const SddmmArgs a)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const int c = blockIdx.x;
    const int e0 = a.bnd[c].y, n = a.bnd[c + 1].y - e0;
    if (a.K / vec_elems(DTB) >= G * NV) sddmm_warp_chunk<DTA, DTB, G, NV, U, true>(a, ring_smem, e0, n);
    else sddmm_warp_chunk<DTA, DTB, G, NV, U, false>(a, ring_smem, e0, n);
}

template <int DTA, int DTB, int G, int NV, int U>
cudaError_t launch_sddmm_warp_shape(const SddmmArgs& a, cudaStream_t s)
{
    const void* fn = (const void*)&k_sddmm_warp<DTA, DTB, G, NV, U>;
    constexpr int smem = SddmmWarp<DTA, DTB, G, NV, U>::BYTES;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks), dim3(32), args, smem, s);
}

// Rows of nv vectors (the last one partial), copied CB bytes at a time.
template <int DTA, int DTB, int G, int NV, int U, int CB>
cudaError_t launch_sddmm_part_shape(const SddmmArgs& a, cudaStream_t s)
{
    const void* fn = (const void*)&k_sddmm_warp_part<DTA, DTB, G, NV, U, CB>;
    constexpr int smem = SddmmWarp<DTA, DTB, G, NV, U>::BYTES;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks), dim3(32), args, smem, s);
}

template <int DTA, int DTB, int CB>
cudaError_t launch_sddmm_part_cb(const SddmmArgs& a, cudaStream_t s)
{
    if (a.nchunks <= 0) return cudaSuccess;
    const int nv = (a.K + vec_elems(DTB) - 1) / vec_elems(DTB);
    if (nv <= 4) return launch_sddmm_part_shape<DTA, DTB, 4, 1, 4, CB>(a, s);
    if (nv <= 8) return launch_sddmm_part_shape<DTA, DTB, 4, 2, 4, CB>(a, s);
    if (nv <= 16) return launch_sddmm_part_shape<DTA, DTB, 8, 2, 4, CB>(a, s);
    return launch_sddmm_part_shape<DTA, DTB, 8, 4, 4, CB>(a, s);
}

}  // namespace spk
