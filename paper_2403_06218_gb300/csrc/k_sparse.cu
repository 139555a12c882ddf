// Sparse kernels: CSR SpMM Y = A X with a tall-skinny dense block (Table 1 "SpMM",
// Alg. 1 S1/S3, Alg. 2 S2/S4) and the one-time build of CSR(A^T) that turns the
// A^T products into the same row-oriented kernel.
//
// A sub-warp of G lanes owns one row; each lane gathers a 16-byte slice of every
// X row the row touches (float4 / double2), so G = w / (16 / sizeof(T)) lanes
// cover a block of w columns and narrow blocks put several rows in a warp.  The
// gathers (nnz w sizeof(T) bytes, from L2 for a block that fits there) bound the
// kernel, not the compulsory HBM bytes: 8 TB/s of gathered data and more on
// GB300 where X stays in L2 (uniform 100,000 x 100,000, 10 entries a row, FP32, 64 columns: 256 MB
// gathered in 31 us = 8.3 TB/s; power-law 2M x 1M: 25.5 GB in 3.3 ms).  FP64 is also close to the
// FP64 pipe's rate (2 DFMA/clk/SM).  Every y_ij is accumulated in CSR order with FMA, so the
// result is deterministic.
//
// Long rows (power-law degrees; CSR(A^T) of a matrix with popular columns holds
// rows of up to ~10^6 entries) would leave one warp working long after the rest.
// A plan built once per matrix cuts every row longer than kSpmmChunk entries into
// chunks of kSpmmChunk: one sub-warp per chunk, in the first blocks of the rows' launch, writes a
// partial row, and a second kernel adds each row's partials in chunk order (still deterministic).
#include <climits>

#include "tsvd_internal.cuh"

namespace tsvd {
namespace {

constexpr unsigned kFull = 0xffffffffu;


// VW consecutive values of the SpMM element type, loaded as one vector.
template <typename T, int VW>
struct VecLoad;
template <>
struct VecLoad<double, 2> {
    __device__ static void get(const double* p, double* o) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p));
        o[0] = v.x;
        o[1] = v.y;
    }
    __device__ static void put(double* p, const double* v) {
        p[0] = v[0];
        p[1] = v[1];
    }
};
template <>
struct VecLoad<float, 4> {
    __device__ static void get(const float* p, float* o) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    }
    __device__ static void put(float* p, const float* v) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <typename T>
struct VecLoad<T, 1> {
    __device__ static void get(const T* p, T* o) { o[0] = __ldg(p); }
    __device__ static void put(T* p, const T* v) { p[0] = v[0]; }
};

// One output row y = sum over the entries [beg, end) of a_e x_{col(e)}, written to
// out[0 .. w) (nothing if out is null), by a sub-warp of G lanes: lane sl owns VW consecutive
// columns of each panel of VW G columns.  Each y_ij is accumulated in CSR order with FMA, so the
// result is deterministic.
// FP32: the lanes read G entries' (col, val) at once and pass them around by shuffles, so that
// four gathers are in flight; with one entry's column, value and gather after the other the kernel
// waited for memory (500,000 x 250,000 power-law, 12 M entries, 100 columns: 1.39 ms, now 0.84).
// FP64: one entry after the other; the FP64 pipe bounds that, and the shuffles only delay it
// (100,000 rows of 10 entries, 128 columns: 325 us against 371 us).
template <typename T, int VW, int G>
__device__ inline void spmm_segment(int64_t beg, int64_t end, int64_t n, const int32_t* __restrict__ ci,
                                    const T* __restrict__ va, int w, const T* __restrict__ X, int64_t ldx,
                                    T* __restrict__ out, int* status, int sl) {
    if constexpr (sizeof(T) == 8) {
        if (!out) return;
        for (int c0 = 0; c0 < w; c0 += VW * G) {
            const int col = c0 + VW * sl;
            if (col >= w) continue;  // lanes past the last column of a narrow panel
            const bool full = col + VW <= w;
            T acc[VW];
#pragma unroll
            for (int q = 0; q < VW; ++q) acc[q] = T(0);
            for (int64_t e = beg; e < end; ++e) {
                const int c = __ldg(ci + e);  // read by all G lanes: a broadcast
                const T a = __ldg(va + e);
                if ((uint64_t)(int64_t)c >= (uint64_t)n) {  // skipped, and reported
                    if (sl == 0) atomicOr(&status[kStBadCsr], 1);
                    continue;
                }
                const T* xr = X + (int64_t)c * ldx + col;
                T x[VW];
                if (full) {
                    VecLoad<T, VW>::get(xr, x);
                } else {
#pragma unroll
                    for (int q = 0; q < VW; ++q) x[q] = (col + q < w) ? __ldg(xr + q) : T(0);
                }
#pragma unroll
                for (int q = 0; q < VW; ++q) acc[q] = fma(a, x[q], acc[q]);
            }
#pragma unroll
            for (int q = 0; q < VW; ++q)
                if (col + q < w) out[col + q] = acc[q];
        }
        return;
    }
    int len = (int)min((int64_t)INT_MAX, max((int64_t)0, end - beg));
    if (G < 32) len = __reduce_max_sync(kFull, len);  // the warp's sub-warps stay together
    for (int c0 = 0; c0 < w; c0 += VW * G) {
        const int col = c0 + VW * sl;
        const int have = min(VW, w - col);  // columns of this lane (none or fewer past a panel's end)
        T acc[VW];
#pragma unroll
        for (int q = 0; q < VW; ++q) acc[q] = T(0);
        for (int o = 0; o < len; o += G) {
            int mc = -1;
            T ma = T(0);
            if (beg + o + sl < end) {
                const int64_t e = beg + o + sl;
                mc = __ldg(ci + e);
                ma = __ldg(va + e);
                if ((uint64_t)(int64_t)mc >= (uint64_t)n) {  // skipped, and reported
                    atomicOr(&status[kStBadCsr], 1);
                    mc = -1;
                }
            }
            __syncwarp();
            const int cnt = min(G, len - o);
            for (int t = 0; t < cnt; t += 4) {
                int c[4];
                T a[4], x[4][VW];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    c[u] = __shfl_sync(kFull, mc, t + u, G);
                    a[u] = __shfl_sync(kFull, ma, t + u, G);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const T* xr = X + (int64_t)c[u] * ldx + col;
                    if (c[u] >= 0 && have == VW) {
                        VecLoad<T, VW>::get(xr, x[u]);
                    } else {
#pragma unroll
                        for (int q = 0; q < VW; ++q) x[u][q] = c[u] >= 0 && q < have ? __ldg(xr + q) : T(0);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    // an entry that is not there adds 0 * 0
                    const T v = c[u] >= 0 ? a[u] : T(0);
                    if (t + u < cnt)
#pragma unroll
                        for (int q = 0; q < VW; ++q) acc[q] = fma(v, x[u][q], acc[q]);
                }
            }
        }
        if (!out) continue;
        if (VW * sizeof(T) == 16 && have == VW && (reinterpret_cast<uintptr_t>(out + col) & 15) == 0) {
            VecLoad<T, VW>::put(out + col, acc);
        } else {
#pragma unroll
            for (int q = 0; q < VW; ++q)
                if (q < have) out[col + q] = acc[q];
        }
    }
}

// Sub-warp of G lanes per row or chunk.  The first blocks take the chunks of the rows longer than
// `split` entries (a chunk: entries [rp[row] + j C, min(rp[row + 1], rp[row] + (j + 1) C)), into
// partial[chunk][0 .. w)), so that they run beside the rows; the others the rows up to `split`.
template <typename T, int VW, int G>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 6 : 0) spmm_rows_kernel(int64_t m, int64_t n, const int32_t* __restrict__ rp,
                                                        const int32_t* __restrict__ ci, const T* __restrict__ va,
                                                        int w, const T* __restrict__ X, int64_t ldx,
                                                        T* __restrict__ Y, int64_t ldy, int64_t split,
                                                        int64_t nchunks, const int4* __restrict__ chunks,
                                                        T* __restrict__ partial, int64_t ldp, int* status) {
    constexpr int per = 256 / G;
    const int64_t cb = (nchunks + per - 1) / per;
    const int sl = threadIdx.x % G, sub = threadIdx.x / G;
    int64_t beg = 0, end = 0;
    T* out = nullptr;
    if ((int64_t)blockIdx.x < cb) {
        const int64_t c = (int64_t)blockIdx.x * per + sub;
        if (c < nchunks) {
            const int4 d = chunks[c];
            beg = (int64_t)rp[d.x] + (int64_t)d.y * kSpmmChunk;
            end = min((int64_t)rp[d.x + 1], beg + kSpmmChunk);
            out = partial + c * ldp;
        }
    } else {
        const int64_t row = ((int64_t)blockIdx.x - cb) * per + sub;
        if (row < m) {
            beg = rp[row], end = rp[row + 1];
            if (end - beg <= split)
                out = Y + row * ldy;
            else
                end = beg;
        }
    }
    spmm_segment<T, VW, G>(beg, end, n, ci, va, w, X, ldx, out, status, sl);
}

// Y[row] = sum of the row's chunk partials in chunk order (the first chunk's warp does the row).
template <typename T>
__global__ void __launch_bounds__(256) spmm_chunk_sum_kernel(int64_t nchunks, const int4* __restrict__ chunks,
                                                             int w, const T* __restrict__ partial, int64_t ldp,
                                                             T* __restrict__ Y, int64_t ldy) {
    const int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= nchunks) return;
    const int4 d = chunks[c];
    if (d.y != 0) return;
    for (int col = lane; col < w; col += 32) {
        T acc = T(0);
        for (int t = 0; t < d.z; ++t) acc += partial[(c + t) * ldp + col];
        Y[(int64_t)d.x * ldy + col] = acc;
    }
}

// Plan: chunks of each row longer than kSpmmChunk entries.
__global__ void spmm_plan_count_kernel(int64_t m, const int32_t* __restrict__ rp, int32_t* __restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int64_t len = (int64_t)rp[i + 1] - rp[i];
    cnt[i] = len > kSpmmChunk ? (int32_t)((len + kSpmmChunk - 1) / kSpmmChunk) : 0;
}

__global__ void spmm_plan_fill_kernel(int64_t m, const int32_t* __restrict__ cnt, const int32_t* __restrict__ off,
                                      int4* __restrict__ chunks) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int32_t k = cnt[i];
    for (int32_t j = 0; j < k; ++j) chunks[off[i] + j] = make_int4((int)i, j, k, 0);
}

// ---- CSR transpose ---------------------------------------------------------

// CSR(A^T) is A's entries sorted by column, stably: CSR order lists rows in increasing
// order, so every row of A^T comes out in increasing original row order.  The sort is an
// LSD radix sort of (column, row, value) with up to 9 bits a pass.  What bounds it is
// memory: a pass reads the columns twice and moves 16 bytes an entry each way.  (Scattering
// by atomic cursors and sorting each segment afterwards needed about 190 passes over the
// segments longer than 4,096 entries of a power-law matrix: 42.3 ms for 500,000 x 250,000
// with 12 M entries, against 0.69 ms now; 1 M uniform entries take the same as before.)

// Warp per row: validates the row's extent and columns, writes the row of every entry.
__global__ void csr_expand_kernel(int64_t m, int64_t n, int64_t nnz, const int32_t* __restrict__ rp,
                                  const int32_t* __restrict__ ci, int32_t* __restrict__ rows, int* status) {
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= m) return;
    const int64_t beg = rp[row], end = rp[row + 1];
    if (row == 0 && lane == 0 && beg != 0) atomicOr(&status[kStBadCsr], 1);
    if (row == m - 1 && lane == 0 && end != nnz) atomicOr(&status[kStBadCsr], 1);
    if (beg < 0 || end > nnz || beg > end) {
        if (lane == 0) atomicOr(&status[kStBadCsr], 1);
        return;
    }
    for (int64_t e = beg + lane; e < end; e += 32) {
        if ((uint64_t)(int64_t)ci[e] >= (uint64_t)n) atomicOr(&status[kStBadCsr], 1);
        rows[e] = (int32_t)row;
    }
}

constexpr int kSortThreads = 256;
constexpr int kSortPer = 16;
constexpr int kSortTile = kSortThreads * kSortPer;  // entries of a CTA
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortMaxBits = 9;
constexpr int kSortMaxDigits = 1 << kSortMaxBits;

// hist[d * tiles + tile]: entries of the tile whose digit is d.
__global__ void __launch_bounds__(kSortThreads) sort_hist_kernel(int64_t nnz, const int32_t* __restrict__ key,
                                                                 int shift, int digits, int64_t tiles,
                                                                 int32_t* __restrict__ hist) {
    __shared__ int cnt[kSortMaxDigits];
    for (int d = threadIdx.x; d < digits; d += kSortThreads) cnt[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll
    for (int i = 0; i < kSortPer; ++i) {
        const int64_t e = base + i * kSortThreads + threadIdx.x;
        if (e < nnz) atomicAdd(&cnt[(key[e] >> shift) & (digits - 1)], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < digits; d += kSortThreads) hist[d * tiles + blockIdx.x] = cnt[d];
}

// One pass: the tile's entries, ranked stably by digit within the tile (each warp ranks
// 512 consecutive entries, 32 at a time, by matching lanes), are put in digit order in
// shared memory and written from there, so each digit's run is one contiguous store.
template <typename T>
__global__ void __launch_bounds__(kSortThreads)
    sort_scatter_kernel(int64_t nnz, const int32_t* __restrict__ key, const int32_t* __restrict__ row,
                        const T* __restrict__ val, int shift, int digits, int64_t tiles,
                        const int32_t* __restrict__ offs, int32_t* __restrict__ okey, int32_t* __restrict__ orow,
                        T* __restrict__ oval) {
    extern __shared__ __align__(16) unsigned char sort_sm[];
    T* sval = reinterpret_cast<T*>(sort_sm);
    int32_t* skey = reinterpret_cast<int32_t*>(sval + kSortTile);
    int32_t* srow = skey + kSortTile;
    int(*cnt)[kSortMaxDigits] = reinterpret_cast<int(*)[kSortMaxDigits]>(srow + kSortTile);  // [warp][digit]
    __shared__ int start[kSortMaxDigits], gofs[kSortMaxDigits], wsum[kSortWarps];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int d = tid; d < kSortWarps * kSortMaxDigits; d += kSortThreads) (&cnt[0][0])[d] = 0;
    for (int d = tid; d < digits; d += kSortThreads) gofs[d] = offs[d * tiles + blockIdx.x];
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile, wbase = base + warp * (32 * kSortPer);
    int32_t k[kSortPer];
    int loc[kSortPer];
#pragma unroll
    for (int i = 0; i < kSortPer; ++i) {
        const int64_t e = wbase + i * 32 + lane;
        k[i] = e < nnz ? key[e] : 0;
    }
#pragma unroll
    for (int i = 0; i < kSortPer; ++i) {
        const bool in = wbase + i * 32 + lane < nnz;
        const unsigned act = __ballot_sync(kFull, in);
        if (in) {
            const int d = (k[i] >> shift) & (digits - 1);
            const unsigned peers = __match_any_sync(act, d);
            const int before = __popc(peers & ((1u << lane) - 1u));
            loc[i] = cnt[warp][d] + before;
            __syncwarp(act);
            if (before == 0) cnt[warp][d] += __popc(peers);
        }
        __syncwarp();
    }
    __syncthreads();
    // per digit: exclusive sums over the warps, then over the digits (two a thread)
    int tot[kSortMaxDigits / kSortThreads];
    int run = 0;
#pragma unroll
    for (int j = 0; j < kSortMaxDigits / kSortThreads; ++j) {
        const int d = tid * (kSortMaxDigits / kSortThreads) + j;
        int acc = 0;
        for (int w = 0; w < kSortWarps; ++w) {
            const int c = cnt[w][d];
            cnt[w][d] = acc;
            acc += c;
        }
        tot[j] = run;
        run += acc;
    }
    int inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int woff = 0;
    for (int w = 0; w < warp; ++w) woff += wsum[w];
#pragma unroll
    for (int j = 0; j < kSortMaxDigits / kSortThreads; ++j)
        start[tid * (kSortMaxDigits / kSortThreads) + j] = woff + inc - run + tot[j];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortPer; ++i) {
        const int64_t e = wbase + i * 32 + lane;
        if (e < nnz) {
            const int d = (k[i] >> shift) & (digits - 1);
            const int pos = start[d] + cnt[warp][d] + loc[i];
            skey[pos] = k[i];
            srow[pos] = row[e];
            sval[pos] = val[e];
        }
    }
    __syncthreads();
    const int count = (int)min((int64_t)kSortTile, nnz - base);
    for (int i = tid; i < count; i += kSortThreads) {
        const int32_t kk = skey[i];
        const int d = (kk >> shift) & (digits - 1);
        const int64_t o = (int64_t)gofs[d] + (i - start[d]);
        okey[o] = kk;
        orow[o] = srow[i];
        oval[o] = sval[i];
    }
}

template <typename T>
constexpr size_t sort_smem() {
    return (sizeof(T) + 2 * sizeof(int32_t)) * kSortTile + sizeof(int) * kSortWarps * kSortMaxDigits;
}

// trp[c] = the first sorted position whose column is at least c (c <= n).
__global__ void csr_rowptr_kernel(int64_t n, int64_t nnz, const int32_t* __restrict__ key, int32_t* __restrict__ trp) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c > n) return;
    int64_t lo = 0, hi = nnz;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (key[mid] < c)
            lo = mid + 1;
        else
            hi = mid;
    }
    trp[c] = (int32_t)lo;
}

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;

// Exclusive scan of a tile of cnt into out, tile total into bsum.
__global__ void __launch_bounds__(kScanThreads) scan_tile_kernel(int64_t n, const int32_t* __restrict__ cnt,
                                                                 int32_t* __restrict__ out,
                                                                 int32_t* __restrict__ bsum) {
    __shared__ int32_t warp_tot[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
    int32_t v[kScanPer];
    int32_t run = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        const int64_t idx = base + i;
        v[i] = idx < n ? cnt[idx] : 0;
        const int32_t t = v[i];
        v[i] = run;
        run += t;
    }
    // inclusive warp scan of per-thread totals
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    int32_t woff = 0;
    for (int i = 0; i < warp; ++i) woff += warp_tot[i];
    const int32_t toff = woff + inc - run;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        const int64_t idx = base + i;
        if (idx < n) out[idx] = v[i] + toff;
    }
    if (threadIdx.x == kScanThreads - 1) bsum[blockIdx.x] = woff + inc;
}

// Single CTA: exclusive scan of the tile totals in place (sequential carry over chunks).
__global__ void __launch_bounds__(1024) scan_sums_kernel(int64_t nb, int32_t* __restrict__ bsum) {
    __shared__ int32_t wt[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t c0 = 0; c0 < nb; c0 += 1024) {
        const int64_t idx = c0 + threadIdx.x;
        const int32_t x = idx < nb ? bsum[idx] : 0;
        int32_t inc = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wt[warp] = inc;
        __syncthreads();
        int32_t woff = 0;
        for (int i = 0; i < warp; ++i) woff += wt[i];
        const int32_t c = carry;
        if (idx < nb) bsum[idx] = c + woff + inc - x;
        __syncthreads();
        if (threadIdx.x == 1023) carry = c + woff + inc;
        __syncthreads();
    }
}

__global__ void scan_add_kernel(int64_t n, int32_t* __restrict__ out, const int32_t* __restrict__ bsum) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += bsum[i / kScanTile];
}

__global__ void to_float_kernel(int64_t n, const double* __restrict__ x, float* __restrict__ y) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

}  // namespace

cudaError_t convert_to_float(tsvd_handle* h, int64_t n, const double* x, float* y, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    h->launches++;
    to_float_kernel<<<(unsigned)blocks, 256, 0, st>>>(n, x, y);
    return cudaGetLastError();
}

template <typename T, int VW, int G>
static void spmm_launch_all(int64_t m, int64_t n, const int32_t* rp, const int32_t* ci, const T* va, int w, const T* X,
                            int64_t ldx, T* Y, int64_t ldy, const SpmmPlan* plan, int* status, cudaStream_t st) {
    const bool split = plan && plan->nchunks > 0;
    const int64_t per_block = 256 / G, nchunks = split ? plan->nchunks : 0;
    T* part = split ? static_cast<T*>(plan->partial) : nullptr;
    const int64_t ldp = spmm_partial_ld(w);
    const int64_t blocks = (m + per_block - 1) / per_block + (nchunks + per_block - 1) / per_block;
    spmm_rows_kernel<T, VW, G><<<(unsigned)blocks, 256, 0, st>>>(
        m, n, rp, ci, va, w, X, ldx, Y, ldy, split ? (int64_t)kSpmmChunk : INT64_MAX, nchunks,
        split ? plan->chunks : nullptr, part, ldp, status);
    if (!split) return;
    spmm_chunk_sum_kernel<T><<<(unsigned)((plan->nchunks + 7) / 8), 256, 0, st>>>(plan->nchunks, plan->chunks, w,
                                                                                  part, ldp, Y, ldy);
}

// Lanes per row: enough 16-byte slices to cover w, at most a warp (wider blocks loop over panels).
template <typename T, int VW>
static void spmm_dispatch(int64_t m, int64_t n, const int32_t* rp, const int32_t* ci, const T* va, int w, const T* X,
                          int64_t ldx, T* Y, int64_t ldy, const SpmmPlan* plan, int* status, cudaStream_t st) {
    const int slices = (w + VW - 1) / VW;
    if (slices <= 4)
        spmm_launch_all<T, VW, 4>(m, n, rp, ci, va, w, X, ldx, Y, ldy, plan, status, st);
    else if (slices <= 8)
        spmm_launch_all<T, VW, 8>(m, n, rp, ci, va, w, X, ldx, Y, ldy, plan, status, st);
    else if (slices <= 16)
        spmm_launch_all<T, VW, 16>(m, n, rp, ci, va, w, X, ldx, Y, ldy, plan, status, st);
    else
        spmm_launch_all<T, VW, 32>(m, n, rp, ci, va, w, X, ldx, Y, ldy, plan, status, st);
}

template <typename T>
cudaError_t launch_spmm(tsvd_handle* h, int64_t m, int64_t n, int64_t nnz, const int32_t* row_ptr,
                        const int32_t* col_idx, const T* val, int w, const T* X, int64_t ldx, T* Y,
                        int64_t ldy, int* status, cudaStream_t st, const SpmmPlan* plan) {
    if (m == 0 || w == 0) return cudaSuccess;
    if (plan && plan->nchunks > 0 && w > plan->wmax) return cudaErrorInvalidValue;
    // compulsory traffic: the CSR arrays, X and Y once each
    const double es = (double)sizeof(T);
    ProfScope prof(h, TSVD_K_APROD, 2.0 * nnz * w,
                   (4.0 + es) * nnz + 4.0 * (m + 1) + es * (double)n * w + es * (double)m * w, st);
    // 16-byte gathers need 16-byte aligned X rows
    const bool v16 = (ldx * sizeof(T)) % 16 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    h->launches += (plan && plan->nchunks > 0) ? 2 : 1;
    if (v16)
        spmm_dispatch<T, 16 / sizeof(T)>(m, n, row_ptr, col_idx, val, w, X, ldx, Y, ldy, plan, status, st);
    else
        spmm_dispatch<T, 1>(m, n, row_ptr, col_idx, val, w, X, ldx, Y, ldy, plan, status, st);
    return cudaGetLastError();
}

size_t spmm_plan_ws(int64_t m, int64_t nnz, int wmax, size_t elem) {
    const int64_t maxc = spmm_max_chunks(nnz);
    Arena ar;
    ar.take<int32_t>(m + 1);                                     // chunks per row
    ar.take<int32_t>(m + 1);                                     // their exclusive scan
    ar.take<int32_t>((m + kScanTile - 1) / kScanTile + 1);       // tile sums
    ar.take<int4>(maxc + 1);                                     // chunk descriptors
    ar.take<char>(elem * (size_t)(maxc + 1) * spmm_partial_ld(wmax));  // partial rows
    return ar.off;
}

int spmm_plan(tsvd_handle* h, int64_t m, int64_t nnz, const int32_t* rp, int wmax, size_t elem, Arena& ar,
              SpmmPlan* plan, cudaStream_t st) {
    const int64_t maxc = spmm_max_chunks(nnz);
    int32_t* cnt = ar.take<int32_t>(m + 1);
    int32_t* off = ar.take<int32_t>(m + 1);
    int32_t* bsum = ar.take<int32_t>((m + kScanTile - 1) / kScanTile + 1);
    int4* chunks = ar.take<int4>(maxc + 1);
    void* partial = ar.take<char>(elem * (size_t)(maxc + 1) * spmm_partial_ld(wmax));
    if (!ar.fits()) return TSVD_ERR_WORKSPACE;
    plan->nchunks = 0;
    plan->chunks = chunks;
    plan->partial = partial;
    plan->wmax = wmax;
    if (m == 0 || nnz <= kSpmmChunk) return TSVD_OK;
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 0.0, st);
    const int64_t nb = (m + kScanTile - 1) / kScanTile;
    h->launches += 5;
    spmm_plan_count_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(m, rp, cnt);
    scan_tile_kernel<<<(unsigned)nb, kScanThreads, 0, st>>>(m, cnt, off, bsum);
    scan_sums_kernel<<<1, 1024, 0, st>>>(nb, bsum);
    scan_add_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(m, off, bsum);
    spmm_plan_fill_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(m, cnt, off, chunks);
    TSVD_TRY_CUDA(cudaGetLastError());
    // number of chunks = off[m-1] + cnt[m-1]
    int32_t last[2] = {0, 0};
    TSVD_TRY_CUDA(cudaMemcpyAsync(&last[0], off + (m - 1), sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TSVD_TRY_CUDA(cudaMemcpyAsync(&last[1], cnt + (m - 1), sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TSVD_TRY_CUDA(cudaStreamSynchronize(st));
    plan->nchunks = (int64_t)last[0] + last[1];
    if (plan->nchunks > maxc) return TSVD_ERR_INVALID_ARG;  // row_ptr inconsistent with nnz
    return TSVD_OK;
}

template cudaError_t launch_spmm<double>(tsvd_handle*, int64_t, int64_t, int64_t, const int32_t*, const int32_t*,
                                         const double*, int, const double*, int64_t, double*, int64_t, int*,
                                         cudaStream_t, const SpmmPlan*);
template cudaError_t launch_spmm<float>(tsvd_handle*, int64_t, int64_t, int64_t, const int32_t*, const int32_t*,
                                        const float*, int, const float*, int64_t, float*, int64_t, int*,
                                        cudaStream_t, const SpmmPlan*);

namespace {

// Passes of the column sort and the bits of each (n - 1 has `bits` bits).
struct SortPlan {
    int passes, bits;
    int64_t tiles, hist;  // CTAs of a pass, histogram entries of the widest
};
SortPlan sort_plan(int64_t n, int64_t nnz) {
    SortPlan p;
    int bits = 1;
    while (bits < 31 && (int64_t(1) << bits) < n) ++bits;
    p.passes = (bits + kSortMaxBits - 1) / kSortMaxBits;
    p.bits = (bits + p.passes - 1) / p.passes;
    p.tiles = (nnz + kSortTile - 1) / kSortTile;
    p.hist = p.tiles << p.bits;
    return p;
}

// Scratch of the sort, carved identically by the sizing and the run.
struct SortBufs {
    int32_t *key[2], *row[2], *hist, *offs, *bsum;
    void* val;
};
SortBufs carve_sort(Arena& ar, const SortPlan& p, int64_t nnz) {
    SortBufs b{};
    for (int i = 0; i < 2; ++i) {
        b.key[i] = ar.take<int32_t>(nnz);
        b.row[i] = ar.take<int32_t>(nnz);
    }
    b.val = ar.take<double>(nnz);
    b.hist = ar.take<int32_t>(p.hist);
    b.offs = ar.take<int32_t>(p.hist);
    b.bsum = ar.take<int32_t>((p.hist + kScanTile - 1) / kScanTile + 1);
    return b;
}

}  // namespace

size_t csr_transpose_ws(int64_t m, int64_t n, int64_t nnz) {
    (void)m;
    Arena ar;
    carve_sort(ar, sort_plan(n, nnz), nnz);
    return ar.off;
}

template <typename T>
int csr_transpose(tsvd_handle* h, int64_t m, int64_t n, int64_t nnz, const int32_t* row_ptr,
                  const int32_t* col_idx, const T* val, int32_t* t_row_ptr, int32_t* t_col_idx,
                  T* t_val, Arena& ar, int* status, cudaStream_t st) {
    const SortPlan p = sort_plan(n, nnz);
    const SortBufs b = carve_sort(ar, p, nnz);
    if (!ar.fits()) return TSVD_ERR_WORKSPACE;
    static thread_local int configured = -1;
    if (configured != h->device) {
        TSVD_TRY_CUDA(cudaFuncSetAttribute(sort_scatter_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sort_smem<T>()));
        configured = h->device;
    }
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 0.0, st);
    if (m > 0) {
        h->launches++;
        csr_expand_kernel<<<(unsigned)((m + 7) / 8), 256, 0, st>>>(m, n, nnz, row_ptr, col_idx, b.row[0], status);
        TSVD_TRY_CUDA(cudaGetLastError());
    }
    int hs[kStCount];
    TSVD_TRY(read_status(st, status, hs));
    if (hs[kStBadCsr]) return TSVD_ERR_INVALID_ARG;
    const int32_t* key = col_idx;
    if (m > 0 && nnz > 0) {
        // the last pass writes the outputs; before it, rows and values alternate between the
        // outputs and the scratch
        const int digits = 1 << p.bits;
        const int64_t nb = (p.hist + kScanTile - 1) / kScanTile;
        const int32_t* row = b.row[0];
        const T* v = val;
        for (int i = 0; i < p.passes; ++i) {
            const bool to_out = (p.passes - 1 - i) % 2 == 0;
            int32_t* orow = to_out ? t_col_idx : b.row[1];
            T* oval = to_out ? t_val : static_cast<T*>(b.val);
            int32_t* okey = b.key[i & 1];
            h->launches += 5;
            sort_hist_kernel<<<(unsigned)p.tiles, kSortThreads, 0, st>>>(nnz, key, i * p.bits, digits, p.tiles, b.hist);
            scan_tile_kernel<<<(unsigned)nb, kScanThreads, 0, st>>>(p.hist, b.hist, b.offs, b.bsum);
            scan_sums_kernel<<<1, 1024, 0, st>>>(nb, b.bsum);
            scan_add_kernel<<<(unsigned)((p.hist + 255) / 256), 256, 0, st>>>(p.hist, b.offs, b.bsum);
            sort_scatter_kernel<T><<<(unsigned)p.tiles, kSortThreads, sort_smem<T>(), st>>>(
                nnz, key, row, v, i * p.bits, digits, p.tiles, b.offs, okey, orow, oval);
            TSVD_TRY_CUDA(cudaGetLastError());
            key = okey;
            row = orow;
            v = oval;
        }
    }
    h->launches++;
    csr_rowptr_kernel<<<(unsigned)((n + 256) / 256), 256, 0, st>>>(n, m > 0 ? nnz : 0, key, t_row_ptr);
    TSVD_TRY_CUDA(cudaGetLastError());
    return TSVD_OK;
}

template int csr_transpose<double>(tsvd_handle*, int64_t, int64_t, int64_t, const int32_t*, const int32_t*,
                                   const double*, int32_t*, int32_t*, double*, Arena&, int*, cudaStream_t);
template int csr_transpose<float>(tsvd_handle*, int64_t, int64_t, int64_t, const int32_t*, const int32_t*,
                                  const float*, int32_t*, int32_t*, float*, Arena&, int*, cudaStream_t);

}  // namespace tsvd
