// Transpose plan: the CSC of S (= CSR of S^T) and the CSR slot of every CSC
// slot.  SpMM^T, the adjoint of SpMM in the pair of Sec. 3.2, runs as an SpMM
// over this pattern with the values gathered through `perm`; the plan depends
// only on the pattern, so it is built once (Sec. 5.1).
//
// Built by a stable least-significant-digit radix sort of (column, nonzero
// index) pairs, 8 bits per pass: per-tile digit histograms, one exclusive scan
// over the digit-major histogram table, and a scatter in which every warp ranks
// its items on its own in index order (ballots and per-warp digit counts), so
// that rows stay ascending inside every column.
#include "common.cuh"

namespace spk {

constexpr int RX_THREADS = 256;
constexpr int RX_ROUNDS = 16;
constexpr int RX_TILE = RX_THREADS * RX_ROUNDS;
constexpr int RX_DIGITS = 256;
constexpr int RX_WARPS = RX_THREADS / 32;

TplanLayout tplan_layout(int64_t M, int64_t N, int64_t nnz, int32_t W)
{
    TplanLayout L;
    size_t off = 0;
    L.colptr = off; off += align256((size_t)(N + 1) * 4);
    L.rowidx = off; off += align256((size_t)nnz * 4 + 4);
    L.perm = off;   off += align256((size_t)nnz * 4 + 4);
    L.sl = sched_layout(N, nnz, W);
    L.sched = off;  off += L.sl.total;
    L.total = off;

    L.passes = radix_passes(N);
    L.nblocks = radix_tiles(nnz);
    size_t t = 0;
    L.keys0 = t; t += align256((size_t)nnz * 4 + 4);
    L.keys1 = t; t += align256((size_t)nnz * 4 + 4);
    L.vals0 = t; t += align256((size_t)nnz * 4 + 4);
    L.vals1 = t; t += align256((size_t)nnz * 4 + 4);
    L.hist = t;  t += align256((size_t)L.nblocks * RX_DIGITS * 4);
    L.scan_tmp = t; t += align256(scan_temp_bytes(L.nblocks * RX_DIGITS));
    L.temp_total = t;
    return L;
}

// hist[d * nblocks + b] = count of digit d in tile b.
__global__ void __launch_bounds__(RX_THREADS) k_rx_hist(const int32_t* __restrict__ keys, int64_t n, int shift,
                                                       int64_t nblocks, int32_t* __restrict__ hist)
{
    __shared__ int32_t h[RX_DIGITS];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RX_TILE + threadIdx.x;
    int32_t key[RX_ROUNDS];
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) {
        const int64_t i = base + (int64_t)k * RX_THREADS;
        key[k] = i < n ? __ldg(keys + i) : 0;
    }
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k)
        if (base + (int64_t)k * RX_THREADS < n) atomicAdd(&h[(key[k] >> shift) & 0xff], 1);
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of one tile.  offs = exclusive scan of hist.  vals_in == NULL
// means the identity (the nonzero index).  A warp ranks 512 consecutive items
// on its own (8 ballots a round find the lanes of equal digit, a counter per
// warp and digit carries over the rounds), so the block meets only to add up
// the warps' counts.  Keys, then values, are put in digit order in shared
// memory and written out in runs of one digit.  All loads of a thread are in
// flight at once; the register limit keeps 3 blocks on an SM.  Per pass of 8.4M
// pairs: 256 items at a time with four block barriers a round and scattered
// writes 91 us; this 42 us.
__global__ void __launch_bounds__(RX_THREADS, 3) k_rx_scatter(const int32_t* __restrict__ keys_in,
                                                             const int32_t* __restrict__ vals_in, int64_t n, int shift,
                                                             int64_t nblocks, const int32_t* __restrict__ offs,
                                                             int32_t* __restrict__ keys_out,
                                                             int32_t* __restrict__ vals_out)
{
    __shared__ int32_t wcnt[RX_WARPS][RX_DIGITS];    // items of a digit in a warp, then where they start in the tile
    __shared__ int32_t base_d[RX_DIGITS];            // global minus tile position of a digit's run
    __shared__ int32_t wsum[RX_WARPS];
    __shared__ int32_t tilebuf[RX_TILE];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t tile = (int64_t)blockIdx.x * RX_TILE;
    const int m = (int)(n - tile < RX_TILE ? n - tile : RX_TILE);    // items of the tile
    const int first = warp * (RX_TILE / RX_WARPS) + lane;            // this thread's items: first + 32 k
    int32_t key[RX_ROUNDS], val[RX_ROUNDS], pos[RX_ROUNDS];
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) key[k] = first + k * 32 < m ? __ldg(keys_in + tile + first + k * 32) : 0;
    if (vals_in) {
#pragma unroll
        for (int k = 0; k < RX_ROUNDS; ++k) val[k] = first + k * 32 < m ? __ldg(vals_in + tile + first + k * 32) : 0;
    } else {
#pragma unroll
        for (int k = 0; k < RX_ROUNDS; ++k) val[k] = (int32_t)tile + first + k * 32;
    }
    const int32_t off = __ldg(offs + (int64_t)tid * nblocks + blockIdx.x);
    for (int d = lane; d < RX_DIGITS; d += 32) wcnt[warp][d] = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) {
        const bool valid = first + k * 32 < m;                       // keys may be anything, negative too
        const int digit = (key[k] >> shift) & 0xff;
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (digit >> b) & 1;
            const unsigned v = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? v : ~v;
        }
        const int before = valid ? wcnt[warp][digit] : 0;
        pos[k] = before + __popc(peers & lt);
        __syncwarp();
        if (valid && (peers & lt) == 0) wcnt[warp][digit] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {   // thread tid owns digit tid
        int32_t run = 0;
#pragma unroll
        for (int w = 0; w < RX_WARPS; ++w) {
            const int32_t c = wcnt[w][tid];
            wcnt[w][tid] = run;
            run += c;
        }
        int32_t incl = run;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int32_t start = incl - run;
        for (int w = 0; w < warp; ++w) start += wsum[w];
#pragma unroll
        for (int w = 0; w < RX_WARPS; ++w) wcnt[w][tid] += start;
        base_d[tid] = off - start;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) {
        if (first + k * 32 >= m) continue;
        pos[k] += wcnt[warp][(key[k] >> shift) & 0xff];
        tilebuf[pos[k]] = key[k];
    }
    __syncthreads();
    // key[k] becomes the destination of the item at place tid + 256 k of the ordered tile
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) {
        const int i = tid + k * RX_THREADS;
        if (i >= m) continue;
        const int32_t q = tilebuf[i];
        key[k] = base_d[(q >> shift) & 0xff] + i;
        keys_out[key[k]] = q;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k)
        if (first + k * 32 < m) tilebuf[pos[k]] = val[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RX_ROUNDS; ++k) {
        const int i = tid + k * RX_THREADS;
        if (i < m) vals_out[key[k]] = tilebuf[i];
    }
}

__global__ void k_iota(int32_t* out, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (int32_t)i;
}

// colptr[j] = number of sorted keys < j.
__global__ void k_colptr(const int32_t* sorted, int64_t nnz, int64_t N, int32_t* colptr)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j > N) return;
    int64_t lo = 0, hi = nnz;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (sorted[mid] < j) lo = mid + 1; else hi = mid;
    }
    colptr[j] = (int32_t)lo;
}

// rowidx[p] = row of CSR slot perm[p], from the COO rows of the schedule.
__global__ void k_rows_gather(const int32_t* __restrict__ coo, const int32_t* __restrict__ perm, int64_t nnz,
                              int32_t* __restrict__ rowidx)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < nnz) rowidx[p] = __ldg(coo + __ldg(perm + p));
}

// The same without a schedule: last r with rowptr[r] <= perm[p].
__global__ void k_rows_of(const int32_t* rowptr, int64_t M, const int32_t* perm, int64_t nnz, int32_t* rowidx)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nnz) return;
    const int32_t e = perm[p];
    int64_t lo = 0, hi = M - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (__ldg(rowptr + mid) <= e) lo = mid; else hi = mid - 1;
    }
    rowidx[p] = (int32_t)lo;
}

// Values of S^T in CSC slot order: out[p] = vals[perm[p]] * vals2[perm[p]]
// (absent factors are 1), the same single FP32 product the SpMM kernels form.
__global__ void k_permute_vals(const int32_t* __restrict__ perm, const float* __restrict__ vals,
                               const float* __restrict__ vals2, int64_t nnz, float* __restrict__ out)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = __ldg(perm + p);
        float v = vals ? __ldg(vals + e) : 1.f;
        if (vals2) v *= __ldg(vals2 + e);
        out[p] = v;
    }
}

cudaError_t launch_permute_vals(const int32_t* perm, const float* vals, const float* vals2, int64_t nnz, float* out,
                                cudaStream_t s)
{
    if (nnz <= 0) return cudaSuccess;
    int64_t blocks = (nnz + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_permute_vals<<<(unsigned)blocks, 256, 0, s>>>(perm, vals, vals2, nnz, out);
    return cudaGetLastError();
}

int radix_passes(int64_t range)
{
    int bits = 0;
    while (bits < 31 && (int64_t(1) << bits) < range) ++bits;
    return (bits + 7) / 8;
}

int64_t radix_tiles(int64_t n) { return n < 1 ? 1 : (n + RX_TILE - 1) / RX_TILE; }

size_t radix_hist_bytes(int64_t n) { return align256((size_t)radix_tiles(n) * RX_DIGITS * 4); }

cudaError_t radix_sort_i32(const int32_t* keys, const int32_t* vals, int64_t n, int passes, int32_t* k0, int32_t* k1,
                           int32_t* v0, int32_t* v1, int32_t* hist, void* scan_tmp, const int32_t** keys_out,
                           const int32_t** vals_out, cudaStream_t s, int32_t* k_last, int32_t* v_last)
{
    const int64_t nblocks = radix_tiles(n);
    const int32_t* kin = keys;
    const int32_t* vin = vals;
    for (int p = 0; n > 0 && p < passes; ++p) {
        int32_t* kout = (p & 1) ? k1 : k0;
        int32_t* vout = (p & 1) ? v1 : v0;
        if (p == passes - 1 && k_last) kout = k_last;
        if (p == passes - 1 && v_last) vout = v_last;
        k_rx_hist<<<(unsigned)nblocks, RX_THREADS, 0, s>>>(kin, n, 8 * p, nblocks, hist);
        cudaError_t err = scan_exclusive_i32(hist, hist, nblocks * RX_DIGITS, scan_tmp, s);
        if (err != cudaSuccess) return err;
        k_rx_scatter<<<(unsigned)nblocks, RX_THREADS, 0, s>>>(kin, vin, n, 8 * p, nblocks, hist, kout, vout);
        kin = kout; vin = vout;
    }
    *keys_out = kin;
    *vals_out = vin;
    return cudaGetLastError();
}

cudaError_t build_transpose(const int32_t* rowptr, const int32_t* colidx, const int32_t* coo_rows, int64_t M,
                            int64_t N, int64_t nnz, char* storage, char* temp, const TplanLayout& L, cudaStream_t s)
{
    int32_t* colptr = reinterpret_cast<int32_t*>(storage + L.colptr);
    int32_t* rowidx = reinterpret_cast<int32_t*>(storage + L.rowidx);
    int32_t* perm = reinterpret_cast<int32_t*>(storage + L.perm);
    int32_t* k0 = reinterpret_cast<int32_t*>(temp + L.keys0);
    int32_t* k1 = reinterpret_cast<int32_t*>(temp + L.keys1);
    int32_t* v0 = reinterpret_cast<int32_t*>(temp + L.vals0);
    int32_t* v1 = reinterpret_cast<int32_t*>(temp + L.vals1);
    int32_t* hist = reinterpret_cast<int32_t*>(temp + L.hist);
    cudaError_t err;

    const int32_t* sorted_keys = colidx;
    const int32_t* sorted_vals = nullptr;
    if (nnz > 0) {
        err = radix_sort_i32(colidx, nullptr, nnz, L.passes, k0, k1, v0, v1, hist, temp + L.scan_tmp, &sorted_keys,
                             &sorted_vals, s, nullptr, perm);
        if (err != cudaSuccess) return err;
    }
    if (nnz > 0 && !sorted_vals) {
        // N <= 1: every key is 0 and the CSR order is already sorted.
        k_iota<<<(unsigned)((nnz + 255) / 256), 256, 0, s>>>(perm, nnz);
        err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    k_colptr<<<(unsigned)((N + 1 + 255) / 256), 256, 0, s>>>(sorted_keys, nnz, N, colptr);
    if (nnz > 0 && coo_rows)
        k_rows_gather<<<(unsigned)((nnz + 255) / 256), 256, 0, s>>>(coo_rows, perm, nnz, rowidx);
    else if (nnz > 0)
        k_rows_of<<<(unsigned)((nnz + 255) / 256), 256, 0, s>>>(rowptr, M, perm, nnz, rowidx);
    return cudaGetLastError();
}

}  // namespace spk
