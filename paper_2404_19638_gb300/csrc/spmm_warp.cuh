// SpMM over the balanced schedule, one warp per chunk (Sec. 3.2, Eq. 2).
//
// A whole warp works on one nonzero at a time: lane l accumulates LB bytes of
// the gathered row (K = 64 FP32: 8 bytes), so a row change is one decision for
// the warp.  With lane groups on chunks of their own, the groups of a warp
// change rows at different nonzeros and run the row writes one after another:
// that took 60 % of the issued instructions on R-MAT scale 20.
//
//   * Gathers: the rows of a batch of U nonzeros are copied into one of two
//     batch slots by 16-byte cp.async, CL lanes a row (CL * 16 bytes cover the
//     K block), while the batch before it is computed.  Copying 16 bytes a
//     lane and reading back RB / 32 keeps the copies wide (32 / CL rows an
//     instruction) whatever a lane consumes.
//   * Index streams: 32 nonzeros a tile, one per lane: coalesced 4-byte loads
//     one tile ahead into registers, so any alignment, second value factor,
//     slot permutation or row scale is handled where the tile is loaded, off
//     the per-nonzero path.  Columns, rows and values of two tiles are staged
//     in shared memory; the ballot of "row differs from the entry before"
//     gives one 32-bit mask of row starts per tile.
//   * Compute: a batch without a row start is U loads and FMAs; any other goes
//     four nonzeros at a time and writes a row where its mask bit is set.
//   * Rows without nonzeros are found from the row pointers, 32 at a time,
//     while the first gathers are in flight, not at the row changes.
//
// Every output element adds its nonzeros in slot order with one FMA each, as
// the row-split and register paths do, so all paths agree bit for bit.
//
// Rows that 16 bytes do not divide (CB < 16) are copied 8 or 4 bytes at a
// time, one per lane, and written element by element; the rest is the same.
// The element path reads each row 4 bytes a lane into registers, one lane
// group a chunk: 171 us against 118 (120,011 x 75,503, 20 nonzeros a
// row, FP32, K = 50).
//
// What bounds it (GB300, R-MAT scale 20, 16.1M nonzeros, K = 64): the
// shared-memory data path, 83 % busy in FP32 (each gathered row is written and
// read once there), and instruction issue for 16-bit rows (the widening).
// Measured, lane-group ring before / this: FP32 0.399 / 0.282 ms, BF16 0.407 /
// 0.220 ms; BF16 K = 128 on the 50M-nonzero bipartite pattern 1.20 / 0.87 ms;
// R-MAT scale 22 BF16 K = 64 0.775 / 0.513 ms.  Register gathers with one
// chunk per lane group and the same row masks: 0.36 / 0.35 ms (too few bytes
// in flight at 28 warps a SM).  Batches of 16 rows up to 256 bytes, 8 above:
// K = 128 FP32 0.49 ms with 8, 0.58 with 16 (half the warps fit); 16-bit
// K = 64 0.289 ms with 8, 0.244 with 16 (per-batch work).
#pragma once
#include "ring.cuh"
#include "rows.cuh"

namespace spk {

// How a finished row is written: FP32 stored, FP32 added to C, or any output
// dtype and mode decided at run time.
enum : int { SPMM_STORE = 0, SPMM_ADD = 1, SPMM_ANY = 2 };

constexpr int64_t SPMM_WARP_MAX_ROW = 65535LL * 512;    // bytes of a row: K blocks of 512, one grid row each

template <int DT, int CL>
struct SpmmWarp {
    static constexpr int RBB = CL * 16;                                       // row bytes of a K block
    static constexpr int U = RBB > 256 ? 8 : 16;                              // nonzeros per batch
    static constexpr int LB = RBB / 32 > dt_bytes(DT) ? RBB / 32 : dt_bytes(DT);  // bytes of a row one lane consumes
    static constexpr int E = LB / dt_bytes(DT);                               // elements one lane accumulates
    static constexpr int EPI = 32 / CL;                                       // rows per copy instruction
    static constexpr int NS = U / EPI;                                        // copies per lane and batch
    static constexpr int BPT = 32 / U;                                        // batches per index tile (even)
    static constexpr int SLOT = U * RBB;
    // two batch slots; two tiles of columns, rows and (each twice) values
    __host__ __device__ static constexpr int bytes(int heads) { return 2 * SLOT + 2 * 32 * 4 * (2 + 2 * heads); }
};

// One lane's columns of a row in FP32: E accumulators, in pairs where E is even.
template <int DT, int E>
struct RowAcc {
    static constexpr int P = (E + 1) / 2;
    f32x2 a[P];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int q = 0; q < P; ++q) a[q] = 0ull;
    }
    // a += s * (E elements of DT at p in shared memory); s holds the value twice
    __device__ __forceinline__ void add(f32x2 s, const unsigned char* p)
    {
        if constexpr (E == 1) {
            Raw<DT, 1> r;
            if constexpr (dt_bytes(DT) == 4) r.w[0] = *reinterpret_cast<const uint32_t*>(p);
            else if constexpr (dt_bytes(DT) == 2) r.w[0] = *reinterpret_cast<const unsigned short*>(p);
            else r.w[0] = *p;
            float f[1];
            unpack_all<DT, 1>(r, f);
            a[0] = __float_as_uint(fmaf(lo2(s), f[0], lo2(a[0])));
        } else if constexpr (DT == DT_F32) {
            if constexpr (E == 2) {
                ffma2(a[0], s, *reinterpret_cast<const f32x2*>(p));
            } else {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
                ffma2(a[0], s, v.x);
                ffma2(a[1], s, v.y);
            }
        } else {
            Raw<DT, E> r;
            constexpr int TB = E * dt_bytes(DT);
            if constexpr (TB == 16) {
                const uint4 v = *reinterpret_cast<const uint4*>(p);
                r.w[0] = v.x; r.w[1] = v.y; r.w[2] = v.z; r.w[3] = v.w;
            } else if constexpr (TB == 8) {
                const uint2 v = *reinterpret_cast<const uint2*>(p);
                r.w[0] = v.x; r.w[1] = v.y;
            } else if constexpr (TB == 4) {
                r.w[0] = *reinterpret_cast<const uint32_t*>(p);
            } else {
                r.w[0] = *reinterpret_cast<const unsigned short*>(p);
            }
            float f[E];
            unpack_all<DT, E>(r, f);
#pragma unroll
            for (int q = 0; q < P; ++q) ffma2(a[q], s, pack2(__float_as_uint(f[2 * q]), __float_as_uint(f[2 * q + 1])));
        }
    }
    __device__ __forceinline__ void get(float (&f)[E]) const
    {
#pragma unroll
        for (int q = 0; q < E; ++q) f[q] = (q & 1) ? hi2(a[q / 2]) : lo2(a[q / 2]);
    }
};

__device__ __forceinline__ int dt_bytes_rt(int dt) { return dt == DT_F32 ? 4 : 2; }

// write_vec at an address instead of an element index of C.
template <int E>
__device__ __forceinline__ void write_vec_at(const SpmmArgs& a, char* p, const float* v)
{
    SpmmArgs b = a;
    b.C = p;
    write_vec<E>(b, 0, v);
}

// The first ne elements of a lane's part of an output row, one by one.
template <int E>
__device__ __forceinline__ void write_some_at(const SpmmArgs& a, char* p, const float* v, int ne, int celt)
{
#pragma unroll
    for (int q = 0; q < E; ++q)
        if (q < ne) write_vec_at<1>(a, p + q * celt, v + q);
}

// A piece of a split row is in its carry slot: the warp that delivers the last
// one adds the pieces in slot order and writes the row.
template <int DT, int CL, int CB>
__device__ __noinline__ void spmm_warp_finish(const SpmmArgs& a, int nkb, int s0, int64_t row)
{
    using W = SpmmWarp<DT, CL>;
    constexpr int E = W::E;
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
    for (int kb = 0; kb < nkb; ++kb) {
        const int c = kb * (W::RBB / dt_bytes(DT)) + lane * E;
        if (lane * W::LB < min(a.K * dt_bytes(DT) - kb * W::RBB, W::RBB)) {
            const int ne = CB < 16 ? min(E, a.K - c) : E;
            float sum[E];
#pragma unroll
            for (int q = 0; q < E; ++q) sum[q] = 0.f;
#pragma unroll 4
            for (int sl = s0; sl < s0 + np; ++sl) {
                float x[E];
                if constexpr (CB < 16) {
#pragma unroll
                    for (int q = 0; q < E; ++q) x[q] = q < ne ? __ldcg(a.carry + (int64_t)sl * a.K + c + q) : 0.f;
                } else {
                    load_elems_cg<DT_F32, E>(a.carry, (int64_t)sl * a.K + c, x);
                }
#pragma unroll
                for (int q = 0; q < E; ++q) sum[q] += x[q];
            }
            if constexpr (CB < 16) {
                const int celt = dt_bytes_rt(a.dtc);
                write_some_at<E>(a, reinterpret_cast<char*>(a.C) + (row * a.ldc + c) * celt, sum, ne, celt);
            } else {
                write_vec<E>(a, row * a.ldc + c, sum);
            }
        }
    }
    __syncwarp();
    if (lane == 0) atomicExch(a.cnt + s0, 0);   // ready for the next launch
}

// FULL: every K block is CL * 16 bytes wide, so every lane copies and accumulates.
// CB: bytes of a copy; below 16, MODE is SPMM_ANY and FULL false.
template <int DT, int CL, int MODE, bool FULL, int CB = 16>
__device__ __forceinline__ void spmm_warp_span(const SpmmArgs& a, unsigned char* wsm, int kb, int nkb, const int2 b0,
                                               const int2 b1, const int4 meta, int head_s0)
{
    using W = SpmmWarp<DT, CL>;
    constexpr int E = W::E, U = W::U, NS = W::NS, BPT = W::BPT;
    const int lane = threadIdx.x & 31;
    const int e0 = b0.y, n = b1.y - b0.y;
    const int rb = min(a.K * dt_bytes(DT) - kb * W::RBB, W::RBB);   // valid bytes of this K block
    const int col0 = kb * (W::RBB / dt_bytes(DT)) + lane * E;       // this lane's first column
    const bool act = (FULL && W::LB * 32 == W::RBB) || lane * W::LB < rb;
    int* const tcol = reinterpret_cast<int*>(wsm + 2 * W::SLOT);    // [2][32]
    int* const trow = tcol + 64;                                    // [2][32]
    f32x2* const tval = reinterpret_cast<f32x2*>(trow + 64);        // [heads][2][32], each value twice
    const f32x2* tval_l = tval;                                     // values of the head this lane's columns are in
    if (a.heads > 1) tval_l += min(col0 / (a.K / a.heads), a.heads - 1) * 64;
    const bool plain = a.vals && !a.vals2 && !a.vperm && a.heads == 1 && DT != DT_E4M3;

    int nc = 0, nr = 0, np = 0;
    float nv = 1.f;
    if (a.vperm && lane < n) np = __ldg(a.vperm + e0 + lane);
    auto load_tile = [&](int i) {                                   // entry i of the chunk into this lane's registers
        if (i >= n) return;
        const int e = e0 + i;
        nc = __ldg(a.colidx + e);
        nr = __ldg(a.rowidx + e);
        if (plain) {
            nv = __ldg(a.vals + e);
        } else if (a.heads == 1) {
            const int vi = a.vperm ? np : e;                        // a permuted slot was loaded one tile before
            nv = a.vals ? __ldg(a.vals + vi) : 1.f;
            if (a.vals2) nv *= __ldg(a.vals2 + vi);
            if (a.vperm && i + 32 < n) np = __ldg(a.vperm + e + 32);
            if constexpr (DT == DT_E4M3) nv *= __ldg(a.b_scale + nc);
        }
    };
    int last = 0;                                                   // row of the last staged entry
    auto stage = [&](int t) -> unsigned {                           // registers -> tile buffer t & 1; row-start mask
        const int o = (t & 1) * 32 + lane, i = 32 * t + lane;
        tcol[o] = nc;
        trow[o] = nr;
        if (a.heads == 1) {
            tval[o] = pack2(__float_as_uint(nv), __float_as_uint(nv));
        } else if (i < n) {
            for (int h = 0; h < a.heads; ++h) {
                const float* v = a.vals + (int64_t)h * a.hstride + e0 + i;
                cpa4(reinterpret_cast<float*>(&tval[h * 64 + o]), v);
                cpa4(reinterpret_cast<float*>(&tval[h * 64 + o]) + 1, v);
            }
        }
        int up = __shfl_up_sync(0xffffffffu, nr, 1);
        if (lane == 0) up = last;
        const unsigned m = __ballot_sync(0xffffffffu, i < n && nr != up);
        last = __shfl_sync(0xffffffffu, nr, 31);
        load_tile(i + 32);
        return m;
    };
    const int sub = lane / CL, vec = lane % CL;
    const bool vin = FULL || vec * 16 < rb;
    const char* __restrict__ Bb = reinterpret_cast<const char*>(a.B) + (int64_t)kb * W::RBB + vec * 16;
    const unsigned ldb_bytes = (unsigned)a.ldb * dt_bytes(DT);
    // rows of one copy instruction next to each other for narrow rows (no bank
    // conflicts), else NS consecutive rows per lane block (one vector load of
    // their columns)
    constexpr bool BLK = NS % 4 == 0;
    const unsigned slot0 = (unsigned)__cvta_generic_to_shared(wsm) + (BLK ? sub * NS : sub) * W::RBB + vec * 16;
    static_assert(CB == 16 || (MODE == SPMM_ANY && !FULL), "");
    const int ne = CB < 16 ? min(E, rb / dt_bytes(DT) - lane * E) : E;      // columns of this lane
    auto issue = [&](const int* cols, unsigned slot, int left) {    // copy a batch of `left` (or U) rows
        if constexpr (CB < 16) {
            constexpr int VPR = W::RBB / CB;                        // copies of a row
            const unsigned dst = slot - (BLK ? sub * NS : sub) * W::RBB - vec * 16 + lane * CB;
            if (left > 0)
                for_const<U * VPR / 32>([&](auto q) {
                    const int r = VPR >= 32 ? q.value / (VPR / 32) : (lane + 32 * q.value) / VPR;
                    const int off = (VPR >= 32 ? lane + 32 * (q.value % (VPR / 32)) : lane % VPR) * CB;
                    const bool in = off < rb && r < left;
                    const char* p = reinterpret_cast<const char*>(a.B) + (int64_t)kb * W::RBB;
                    if (in) p += (size_t)(unsigned)cols[r] * ldb_bytes + off;
                    cpa_part<CB, q.value * 32 * CB>(in, dst, p);
                });
        } else if (left > 0) {
            int j[NS];
            if constexpr (BLK) {
#pragma unroll
                for (int c = 0; c < NS / 4; ++c) {
                    const int4 v = *reinterpret_cast<const int4*>(cols + sub * NS + 4 * c);
                    j[4 * c] = v.x; j[4 * c + 1] = v.y; j[4 * c + 2] = v.z; j[4 * c + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < NS; ++i) j[i] = cols[i * W::EPI + sub];
            }
            constexpr int STEP = BLK ? W::RBB : W::EPI * W::RBB;
            if (FULL && left >= U) {
                for_const<NS>([&](auto i) { cpa16_at<i.value * STEP>(slot, Bb + (size_t)(unsigned)j[i.value] * ldb_bytes); });
            } else {
                for_const<NS>([&](auto i) {
                    cpa16_if<i.value * STEP>(vin && (BLK ? sub * NS + i.value : i.value * W::EPI + sub) < left, slot,
                                             Bb + (size_t)(unsigned)j[i.value] * ldb_bytes);
                });
            }
        }
        cp_async_commit();
    };

    RowAcc<DT, E> acc;
    acc.clear();
    float old[E];
    int piece = meta.x >= 0;                                        // the current row goes to a carry slot
    const int celt = MODE == SPMM_ANY ? dt_bytes_rt(a.dtc) : 4;
    char* const Cl = reinterpret_cast<char*>(a.C) + (int64_t)col0 * celt;
    const int64_t ldc_bytes = a.ldc * celt;
    char* dst = nullptr;                                            // this lane's columns of the current row, in C or its carry slot
    auto open = [&](int row) {                                      // start a row that ends in C
        dst = Cl + row * ldc_bytes;
        if constexpr (MODE == SPMM_ADD)
            if (act) load_elems_cg<DT_F32, E>(dst, 0, old);         // arrives while the row is summed
    };
    auto carry_slot = [&](int slot) { return reinterpret_cast<char*>(a.carry + (int64_t)slot * a.K + col0); };
    auto close = [&]() {                                            // write the current row and clear it
        if (act) {
            float f[E];
            acc.get(f);
            if constexpr (MODE == SPMM_ANY) {
                if constexpr (CB < 16) {
                    if (piece) {
#pragma unroll
                        for (int q = 0; q < E; ++q)
                            if (q < ne) reinterpret_cast<float*>(dst)[q] = f[q];
                    } else {
                        write_some_at<E>(a, dst, f, ne, celt);
                    }
                } else {
                    if (piece) store_elems<DT_F32, E>(dst, 0, f);
                    else write_vec_at<E>(a, dst, f);
                }
            } else {
                if constexpr (MODE == SPMM_ADD) {
                    if (!piece) {
#pragma unroll
                        for (int q = 0; q < E; ++q) f[q] += old[q];
                    }
                }
                store_elems<DT_F32, E>(dst, 0, f);
            }
        }
        piece = 0;
        acc.clear();
    };
    const unsigned char* const read0 = wsm + lane * W::LB;
    auto compute = [&](const unsigned char* slot, int o, unsigned m, int left) {
        const f32x2* sv = tval_l + o;
        auto four = [&](int c) {
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                const ulonglong2 s2 = *reinterpret_cast<const ulonglong2*>(sv + c + q);
                acc.add(s2.x, slot + (c + q) * W::RBB);
                acc.add(s2.y, slot + (c + q + 1) * W::RBB);
            }
        };
        if (m == 0 && left >= U) {
#pragma unroll
            for (int c = 0; c < U; c += 4) four(c);
            return;
        }
        const int* rows = trow + o;
        if (left >= U) {
#pragma unroll 1
            for (int c = 0; c < U; c += 4, m >>= 4) {
                if ((m & 15u) == 0) {
                    four(c);
                    continue;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((m >> q) & 1u) {
                        close();
                        open(rows[c + q]);
                    }
                    acc.add(sv[c + q], slot + (c + q) * W::RBB);
                }
            }
        } else {
#pragma unroll 1
            for (int u = 0; u < left; ++u, m >>= 1) {
                if (m & 1u) {
                    close();
                    open(rows[u]);
                }
                acc.add(sv[u], slot + u * W::RBB);
            }
        }
    };
    auto zero_rows = [&]() {                                        // rows of the chunk without nonzeros
        if (MODE == SPMM_ADD || (MODE == SPMM_ANY && a.accumulate)) return;
        float z[E];
#pragma unroll
        for (int q = 0; q < E; ++q) z[q] = 0.f;
        for (int r0 = b0.x; r0 <= meta.z; r0 += 32) {
            const int r = r0 + lane;
            bool none = false;
            if (r <= meta.z) none = __ldg(a.rowptr + r) == __ldg(a.rowptr + r + 1);
            unsigned zm = __ballot_sync(0xffffffffu, none);
            while (zm) {
                char* p = Cl + (r0 + __ffs(zm) - 1) * ldc_bytes;
                zm &= zm - 1;
                if (!act) continue;
                if constexpr (CB < 16) write_some_at<E>(a, p, z, ne, celt);
                else if constexpr (MODE == SPMM_ANY) store_elems<DT_BF16, E>(p, 0, z);      // BF16 and F16 zeros are the same bits
                else store_elems<DT_F32, E>(p, 0, z);
            }
        }
    };

    if (n <= 0) {
        zero_rows();
        return;
    }
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
        // batch q of the tile is in slot q & 1; the next one is copied before it is waited for
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
            if (left > 0) compute(read0 + (q & 1) * W::SLOT, o + q * U, (m >> (q * U)) & ((1u << U) - 1u), left);
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
    if (meta.x >= 0) spmm_warp_finish<DT, CL, CB>(a, nkb, head_s0, b0.x);
    if (meta.y >= 0) spmm_warp_finish<DT, CL, CB>(a, nkb, meta.y, b1.x);
}

// One warp per CTA and chunk (so that every per-chunk quantity is uniform over
// the CTA and row changes are plain branches), one grid row per K block of
// CL * 16 bytes.
template <int DT, int CL, int MODE, bool FULL, int CB = 16>
__global__ void __launch_bounds__(32) k_spmm_warp(const SpmmArgs a)
{
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const int64_t c = blockIdx.x;
    const int2 b0 = a.bnd[c], b1 = a.bnd[c + 1];
    const int4 m = a.meta[c];
    const int hs0 = (m.x >= 0) ? __ldg(a.head_s0 + c) : -1;
    spmm_warp_span<DT, CL, MODE, FULL, CB>(a, ring_smem, blockIdx.y, gridDim.y, b0, b1, m, hs0);
}

template <int DT, int CL, int CB = 16>
cudaError_t launch_spmm_warp_cl(const SpmmArgs& a, cudaStream_t s)
{
    using W = SpmmWarp<DT, CL>;
    const int rb = a.K * dt_bytes(DT);
    const int nkb = (rb + W::RBB - 1) / W::RBB;
    if (nkb > 65535) return cudaErrorInvalidValue;
    if constexpr (CB < 16) {
        const void* fn = (const void*)&k_spmm_warp<DT, CL, SPMM_ANY, false, CB>;
        const size_t smem = W::bytes(a.heads);
        void* args[] = {(void*)&a};
        return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks, (unsigned)nkb), dim3(32), args, smem, s);
    } else {
    const int mode = a.dtc != DT_F32 ? SPMM_ANY : (a.accumulate ? SPMM_ADD : SPMM_STORE);
    const bool full = rb % W::RBB == 0;
    const void* fn = mode == SPMM_STORE ? (full ? (const void*)&k_spmm_warp<DT, CL, SPMM_STORE, true>
                                                : (const void*)&k_spmm_warp<DT, CL, SPMM_STORE, false>)
                   : mode == SPMM_ADD   ? (full ? (const void*)&k_spmm_warp<DT, CL, SPMM_ADD, true>
                                                : (const void*)&k_spmm_warp<DT, CL, SPMM_ADD, false>)
                                        : (full ? (const void*)&k_spmm_warp<DT, CL, SPMM_ANY, true>
                                                : (const void*)&k_spmm_warp<DT, CL, SPMM_ANY, false>);
    const size_t smem = W::bytes(a.heads);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3((unsigned)a.nchunks, (unsigned)nkb), dim3(32), args, smem, s);
    }
}

// K blocks of the smallest 2^k x 32 bytes that holds a row, at most 512.
template <int DT, int CB = 16>
cudaError_t launch_spmm_warp(SpmmArgs a, cudaStream_t s)
{
    if (a.nchunks <= 0) return cudaSuccess;
    if (!a.vals) a.heads = 1;                            // ones for every head
    const int rb = a.K * dt_bytes(DT);
    if (rb <= 32) return launch_spmm_warp_cl<DT, 2, CB>(a, s);
    if (rb <= 64) return launch_spmm_warp_cl<DT, 4, CB>(a, s);
    if (rb <= 128) return launch_spmm_warp_cl<DT, 8, CB>(a, s);
    if (rb <= 256) return launch_spmm_warp_cl<DT, 16, CB>(a, s);
    return launch_spmm_warp_cl<DT, 32, CB>(a, s);
}

}  // namespace spk
