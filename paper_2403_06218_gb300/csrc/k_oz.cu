// FP64-accurate products on the tensor cores for the FP64 method: the Gram and
// projection products of CholeskyQR2 and CGS-CQR2 (Alg. 4 S1/S4, Alg. 5 S1/S6:
// C = X^T Z), the updates and triangular solves (Alg. 5 S2/S7, Alg. 4 S3/S6:
// Y = beta Y + alpha X M), and the Ritz / restart products (Alg. 2 S7-S9).
// GB300's FP64 pipe issues 2 DFMA/clk/SM; its BF16 tensor cores are about 1500x
// faster, so these products are run as exact integer arithmetic on BF16 digits
// (the exponent-aligned slicing of Ozaki, Ogita, Oishi and Rump, 2012, with the
// fixed-point digits of Ootomo, Ozaki and Yokota, 2024):
//
//  * every row of the left operand A and every column of the right operand B
//    gets one exponent e (the smallest e with |x| < 2^e over that row or
//    column); each entry becomes the 56-bit integer F = round(x 2^(55 - e)),
//    split into 7 balanced base-256 digits d_0..d_6 (F = sum d_p 2^(8(6-p)),
//    |d_p| <= 128).  Digit p is stored as the BF16 value d_p (exact);
//  * the 28 digit products with p + q <= 6 are issued as tcgen05 MMAs (M = 128,
//    K = 16, FP32 accumulators in tensor memory), one accumulator per value of
//    g = p + q (7 accumulators side by side); the products of one A digit plane with
//    several B planes form a single MMA of N up to 256.  Each product is an integer of
//    magnitude <= 2^14 and the group sum T_g adds g + 1 of them per k, so over 256 k
//    (T_0 .. T_3) or 128 k (T_4 .. T_6) it is an integer within 2^24 and every
//    accumulation is exact whatever the tensor core's internal rounding;
//  * after that many k the epilogue converts the accumulators to integers and adds
//    T_0..T_4 into a 64-bit integer (units of 2^-32 of the leading digit
//    product), T_5 and T_6 (rounded to 2^-40) into a 32-bit one, and at the end
//    of its K range writes C = 2^(ea + eb - 46) (hi + lo 2^-8) in FP64.
// Each operand entry is represented to 2^-56 of its row (column) scale 2^e, the
// dropped digit products are below 6.1 K 2^(ea + eb - 56), and the result is
// rounded once to FP64: normwise FP64 accuracy (checked against exact products
// in the CPU tests of the scheme and on the GPU).
//
// Layout: every operand is sliced into 7 BF16 digit planes stored K-block major (oz_off),
// by one of three slicing kernels:
//   rows  the source rows are the stored rows (A = X of X M: one exponent per
//         source row, computed by the warp that slices the row);
//   grow  the same for a basis that gains columns block by block;
//   cols  the source columns are the stored rows (A = X^T and B = Z of X^T Z,
//         B = M of X M: one exponent per source column, from a column-max pass
//         with atomicMax, then a tiled transpose).
// Operands that many products read (a Lanczos basis, a dense A) keep their planes
// in a cache that the owner extends block by block.
// The product kernel (one CTA per SM) is a TMA / tcgen05 pipeline: warp 0 copies the 7
// planes of both operands' K blocks into a ring of 5 to 7 stages, warp 1 owns the tensor
// memory and issues the 11 MMAs of each stage from one thread, the other warps read the
// accumulators.  Work
// units (output tile, 16-wide K block) are split evenly over one wave of CTAs,
// so no CTA runs a third tile while the others idle (314 tiles on 152 SMs would
// take three rounds for 2.07 rounds of work): a tile whose K range lies inside
// one CTA's share is written by its epilogue, the few tiles cut between CTAs
// leave partial tiles that a fix-up kernel adds in CTA order, so the result is
// deterministic.  Every mbarrier wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "tc_ptx.cuh"
#include "tsvd_internal.cuh"

namespace tsvd {
namespace {

using namespace tcx;

constexpr int kOzDig = 7;                                   // digits per operand entry
constexpr int kOzWideDig = 8;                               // of the wide form
constexpr int kOzM = 128;                                   // output rows per tile (TMEM lanes)
constexpr int kOzN = 64;                                    // most output columns per tile
constexpr int kOzBK = 16;                                   // K per stage (one 32-byte row, one MMA)
constexpr int kOzRowB = 2 * kOzBK;
constexpr int kOzPlaneA = kOzM * kOzRowB;                   // 4 KB
constexpr int kOzLowSlots = 4;       // p + q = 0 .. 3: the low group; 4 .. 6 (or 7): the high group
// K blocks of one exact accumulation (every |T_g| <= (g + 1) 2^14 per k stays within 2^24):
// 256 k for T_0 .. T_3, 128 k for the others.  The low chunks end 4 K blocks off the high
// ones, the first one after 12 K blocks (so that a tile's output has 8 to finish in).
constexpr int kOzLowChunk = 16, kOzHighChunk = 8, kOzLowShift = 4;
constexpr int kOzRun = 4;             // K blocks issued for one group before the other takes over
constexpr int kOzFoldChunks = 128;    // high chunks between carries of lo into hi (lo stays below 2^31)
constexpr int kOzFlushChunks = 768;   // high chunks between FP64 flushes of the integer sums (98,304 k)
constexpr int kOzWave = 152;

// Tile shapes: NC columns, D digits, slot p + q at TMEM column (p + q) NC.
template <int NC, int D>
struct OzShape {
    static constexpr int kStageA = D * kOzPlaneA;                    // 28 (32) KB
    static constexpr int kPlaneB = NC * kOzRowB;                     // 2 KB at 64 columns
    static constexpr int kStage = kStageA + D * kPlaneB;
    static constexpr int kStages = D == 7 ? (NC == 64 ? 5 : (NC == 32 ? 6 : 7)) : (NC == 64 ? 4 : (NC == 32 ? 5 : 6));
    static constexpr int kSmem = kStages * kStage + 1024;
    static constexpr int kTmemCols = NC == 64 ? 512 : (NC == 32 ? 256 : 128);
    static constexpr int kEpiWarps = NC == 64 ? 16 : 8;              // NC / 4 or NC / 2 columns a warp
    static constexpr int kThreads = 64 + 32 * kEpiWarps;             // TMA warp, MMA warp, epilogue
};
constexpr int kOzNanExp = 1 << 20;      // exponent of a row holding Inf or NaN
constexpr int kOzZeroExp = -(1 << 20);  // exponent of a zero entry

// ---- digits ------------------------------------------------------------------
__device__ inline int oz_exp(double x) {
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    const int be = (int)((u >> 52) & 0x7FF);
    const uint64_t mant = u & ((1ull << 52) - 1);
    if (be == 0x7FF) return kOzNanExp;
    if (be == 0) return mant == 0 ? kOzZeroExp : (63 - __clzll((long long)mant)) - 1073;
    return be - 1022;
}

__device__ inline int oz_norm_exp(int e) { return e <= kOzZeroExp ? 0 : e; }

// Balanced triangular products (wide form): X M = (X D^-1)(D M), D the powers of two above the
// columns of X.  c: exponent of D at a column from its column maximum (1 for a column of zeros
// or with Inf or NaN); oz_exp_over: exponent of x / 2^c.
__device__ inline int oz_balance(const int* cexp, int64_t k) {
    const int e = cexp ? cexp[k] : 0;
    return e <= kOzZeroExp || e >= kOzNanExp ? 0 : e;
}
__device__ inline int oz_exp_over(double x, int c) {
    const int e = oz_exp(x);
    return e <= kOzZeroExp || e >= kOzNanExp ? e : e - c;
}

// F = round(x 2^(T - e)) (ties away from zero; T = 8 D - 1) plus
// sum_p 128 256^p over the D digits: digit p of F is then byte D - 1 - p of the sum less 128
// (the leading one may need a ninth bit: with 8 digits it is lost, and 128 reads as -128).
template <int D>
__device__ inline unsigned long long oz_biased(double x, int e) {
    constexpr int T = 8 * D - 1;
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    const int be = (int)((u >> 52) & 0x7FF);
    uint64_t m = u & ((1ull << 52) - 1);
    int q = -1074;
    if (be != 0) {
        m |= 1ull << 52;
        q = be - 1075;
    }
    // a row holding Inf or NaN has an exponent that shifts everything out
    const int sh = q + T - e;  // <= T - 53 when |x| < 2^e
    uint64_t F = 0;
    if (sh >= 0)
        F = m << sh;
    else if (sh > -54)
        F = (m + (1ull << (-sh - 1))) >> (-sh);
    if (u >> 63) F = 0ull - F;
    return F + (D == 7 ? 0x80808080808080ull : 0x8080808080808080ull);
}

// Digit p as a float: the byte becomes the low mantissa bits of 2^23.
template <int D>
__device__ inline float oz_digit(unsigned long long w, int p) {
    const int i = D - 1 - p;
    const unsigned half = i < 4 ? (unsigned)w : (unsigned)(w >> 32);
    const unsigned sel = D == 7 && p == 0 ? 0x7432u : 0x7540u | (unsigned)(i & 3);
    return __uint_as_float(__byte_perm(half, 0x4B000000u, sel)) - 8388736.0f;  // 2^23 + 128
}

// Global layout of the digit planes: K-block major, and within a block the very bytes that
// the MMA reads from shared memory.  Element (digit p, stored row r, column k) of an operand
// with Ra allocated stored rows (a multiple of 16) sits at
//   ((k / 16) * D + p) * Ra * 16 + r * 16 + (k % 16, its halves of 8 exchanged in every
//   second group of 4 rows: the 32-byte swizzle),
// so that a TMA box of 128 rows x 7 planes is 56 runs of 512 bytes copied as they are.  (As
// a box of 16 columns, swizzled by the copy, it was 896 runs of 32 bytes, and the copy
// engine's rate of about 1.4 clocks a run bounded the product kernel: 1,344 runs a stage.)
// Columns past K up to the next multiple of 16 hold zeros.
template <int D>
__host__ __device__ inline int64_t oz_off(int64_t Ra, int64_t r, int64_t k, int p) {
    return ((k >> 4) * D + p) * Ra * 16 + r * 16 + ((k & 15) ^ ((r & 4) << 1));
}
__host__ __device__ inline int64_t oz_k16(int64_t K) { return (K + 15) / 16 * 16; }
inline int64_t oz_ra(int64_t rows) { return (rows + 15) / 16 * 16; }

// Stores the digits of (x0, x1) at columns (k, k + 1), k even, of stored row r.  The slicers
// give 8 lanes to the 16 columns of a K block and the 4 groups of 8 to consecutive stored
// rows, so that a warp's store of one digit is 128 contiguous bytes.
template <int D>
__device__ inline void oz_store_pair(__nv_bfloat16* planes, int64_t Ra, int64_t r, int64_t k, double x0, double x1,
                                     int e0, int e1) {
    const unsigned long long a = oz_biased<D>(x0, e0), b = oz_biased<D>(x1, e1);
    __nv_bfloat162* dst = reinterpret_cast<__nv_bfloat162*>(planes + oz_off<D>(Ra, r, k, 0));
#pragma unroll
    for (int p = 0; p < D; ++p) {  // exact: |digit| <= 128; plane step Ra * 16 elements
        float da = oz_digit<D>(a, p), db = oz_digit<D>(b, p);
        if (D == 8 && p == 0) {  // the leading digit has the entry's sign
            da = x0 > 0.0 ? fabsf(da) : da;
            db = x1 > 0.0 ? fabsf(db) : db;
        }
        dst[p * Ra * 8] = __floats2bfloat162_rn(da, db);
    }
}
template <int D>
__device__ inline void oz_store_pair(__nv_bfloat16* planes, int64_t Ra, int64_t r, int64_t k, double x0, double x1,
                                     int e) {
    oz_store_pair<D>(planes, Ra, r, k, x0, x1, e, e);
}

// Rows slicer: columns [c0, c1) of S (R rows, lds) -> columns [c0, c1) of stored row i, zeros
// from c1 to the next multiple of 16; G lanes a row: 8, or 32 where the rows are few (512 x 512
// took 45 us with 8, 4,096 lanes in all).
// GROW false (c0 = 0): the exponent of a row's largest entry.  GROW true, for a matrix that
// gains columns (a Lanczos basis): one above it when it is set (at c0 = 0, or when a later
// entry does not fit it: the row's earlier columns are then sliced again), so that new
// columns rarely raise it.  That keeps 55 bits below the row's largest entry; one exponent
// for all rows of an orthonormal basis kept about log2(R) / 2 bits fewer.
// BAL: the entries over the powers of two above their columns (cexp, oz_balance).
// Bound by the 14 (16) bytes written and 8 read an entry (the digits are read again from
// cache where a row group fits it): 100,000 x 64 in 27 us = 5.2 TB/s.
template <int D, bool GROW, int G, bool BAL = false>
__global__ void __launch_bounds__(256, 4) oz_slice_rows_kernel(int64_t R, int64_t c0, int64_t c1,
                                                            const double* __restrict__ S, int64_t lds,
                                                            __nv_bfloat16* __restrict__ planes, int64_t Ra,
                                                            int* __restrict__ eexp, const int* __restrict__ cexp) {
    const int sl = threadIdx.x % G;
    const int64_t ng = (int64_t)gridDim.x * (blockDim.x / G);
    const int64_t rounds = (R + ng - 1) / ng;  // the same for every lane: the shuffles need them all
    const int64_t a1 = oz_k16(c1);
    for (int64_t t = 0; t < rounds; ++t) {
        const int64_t i = t * ng + (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
        const bool in = i < R;
        const double* src = S + i * lds;
        int e = kOzZeroExp;
        if (in) {
#pragma unroll 4
            for (int64_t k = c0 + sl; k < c1; k += G)
                e = max(e, BAL ? oz_exp_over(src[k], oz_balance(cexp, k)) : oz_exp(src[k]));
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        int64_t k0 = 0;
        if (GROW) {
            int old = in && sl == 0 && c0 > 0 ? eexp[i] : kOzZeroExp;
            old = __shfl_sync(0xffffffffu, old, (threadIdx.x & 31) & ~(G - 1));
            // (a row of zeros keeps the exponent of zero, which any entry exceeds)
            const bool set = c0 == 0 || e > old;
            e = !set ? old : (e >= kOzNanExp || e <= kOzZeroExp ? e : e + 1);
            if (!set) k0 = c0 & ~int64_t(15);
            if (in && set && sl == 0) eexp[i] = e;
        } else {
            e = oz_norm_exp(e);
            if (in && sl == 0) eexp[i] = e;
        }
        if (!in) continue;
        for (int64_t k = k0 + 2 * sl; k < a1; k += 2 * G) {
            const int s0 = BAL && k < c1 ? oz_balance(cexp, k) : 0, s1 = BAL && k + 1 < c1 ? oz_balance(cexp, k + 1) : 0;
            oz_store_pair<D>(planes, Ra, i, k, k < c1 ? src[k] : 0.0, k + 1 < c1 ? src[k + 1] : 0.0, e + s0, e + s1);
        }
    }
}

// Exponent arrays start below every exponent (memset of 0x80 bytes) and grow by atomicMax.
constexpr int kOzUnset = 0x80;

// Column maxima of the exponents of S (K x R, lds); upper: entries with k > j are zero.
__global__ void __launch_bounds__(256) oz_colmax_kernel(int64_t K, int64_t R, const double* __restrict__ S,
                                                        int64_t lds, int upper, int64_t rows_per,
                                                        int* __restrict__ eexp) {
    __shared__ int red[8][33];
    const int64_t j = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int64_t k0 = (int64_t)blockIdx.y * rows_per, k1 = min(K, k0 + rows_per);
    int e = kOzZeroExp;
    if (j < R) {
#pragma unroll 8
        for (int64_t k = k0 + threadIdx.y; k < k1; k += 8)
            if (!(upper && k > j)) e = max(e, oz_exp(S[k * lds + j]));
    }
    red[threadIdx.y][threadIdx.x] = e;
    __syncthreads();
    if (threadIdx.y == 0 && j < R) {
#pragma unroll
        for (int y = 1; y < 8; ++y) e = max(e, red[y][threadIdx.x]);
        atomicMax(&eexp[j], e);
    }
}

// Row and column maxima of the exponents of S (M x N, lds) in one read: a block of 128 rows
// x 256 columns, one thread a column, a row's maximum by a warp reduction.
__global__ void __launch_bounds__(256) oz_max_both_kernel(int64_t M, int64_t N, const double* __restrict__ S,
                                                          int64_t lds, int* __restrict__ rexp,
                                                          int* __restrict__ cexp) {
    __shared__ int rmax[128];
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x, i0 = (int64_t)blockIdx.y * 128;
    const int rows = (int)min((int64_t)128, M - i0);
    if (threadIdx.x < 128) rmax[threadIdx.x] = kOzZeroExp;
    __syncthreads();
    int c = kOzZeroExp;
    const double* src = S + i0 * lds + j;
#pragma unroll 8
    for (int r = 0; r < rows; ++r) {
        const int e = j < N ? oz_exp(src[(int64_t)r * lds]) : kOzZeroExp;
        c = max(c, e);
        const int w = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0) atomicMax(&rmax[r], w);
    }
    if (j < N) atomicMax(&cexp[j], c);
    __syncthreads();
    if ((int)threadIdx.x < rows) atomicMax(&rexp[i0 + threadIdx.x], rmax[threadIdx.x]);
}

// Slices a 64 x 64 tile of S (M x N, lds) from shared memory (row stride 65): its rows into
// the rows layout (stored row i, K = N) and its columns into the cols layout (stored row
// j, K = M), or the columns alone.
template <int D, bool ROWS>
__device__ inline void oz_slice_tile(const double (*tile)[65], int64_t i0, int64_t j0, int64_t M, int64_t N,
                                     const int* __restrict__ rexp, const int* __restrict__ cexp,
                                     __nv_bfloat16* __restrict__ rplanes, int64_t rRa,
                                     __nv_bfloat16* __restrict__ cplanes, int64_t cRa, int64_t c0) {
    const int warp = threadIdx.x >> 5, pr = 2 * (threadIdx.x & 7), sub = (threadIdx.x & 31) >> 3;
#pragma unroll 1
    for (int u = warp; u < 64; u += 8) {  // K block u / 16, 4 stored rows
        const int kb = (u >> 4) * 16 + pr, q = (u & 15) * 4 + sub;
        if (ROWS && i0 + q < M && j0 + kb < oz_k16(N))
            oz_store_pair<D>(rplanes, rRa, i0 + q, j0 + kb, tile[q][kb], tile[q][kb + 1],
                             oz_norm_exp(rexp[i0 + q]));
        if (j0 + q < N && i0 + kb < oz_k16(M))
            oz_store_pair<D>(cplanes, cRa, c0 + j0 + q, i0 + kb, tile[kb][q], tile[kb + 1][q],
                             oz_norm_exp(cexp[j0 + q]));
    }
}

// Both layouts of a matrix in one read (a dense A, whose products need both): with the one
// read of oz_max_both that is 16 bytes read and 28 written an entry, against 32 and 28 by
// the single-layout slicers.
template <int D>
__global__ void __launch_bounds__(256)
    oz_slice_both_kernel(int64_t M, int64_t N, const double* __restrict__ S, int64_t lds,
                         const int* __restrict__ rexp, const int* __restrict__ cexp,
                         __nv_bfloat16* __restrict__ rplanes, int64_t rRa, __nv_bfloat16* __restrict__ cplanes,
                         int64_t cRa) {
    __shared__ double tile[64][65];
    const int64_t i0 = (int64_t)blockIdx.y * 64, j0 = (int64_t)blockIdx.x * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
#pragma unroll
    for (int r = ty; r < 64; r += 4)
        tile[r][tx] = i0 + r < M && j0 + tx < N ? S[(i0 + r) * lds + j0 + tx] : 0.0;
    __syncthreads();
    oz_slice_tile<D, true>(tile, i0, j0, M, N, rexp, cexp, rplanes, rRa, cplanes, cRa, 0);
}

// Cols slicer: column j of S (K x R, lds) -> stored row r0 + j, tiles of 64 k x 64 j, zeros
// past K up to the next multiple of 16.
template <int D>
__global__ void __launch_bounds__(256) oz_slice_cols_kernel(int64_t K, int64_t R, const double* __restrict__ S,
                                                            int64_t lds, int upper, const int* __restrict__ eexp,
                                                            __nv_bfloat16* __restrict__ planes, int64_t Ra,
                                                            int64_t r0) {
    __shared__ double tile[64][65];
    const int64_t k0 = (int64_t)blockIdx.x * 64, j0 = (int64_t)blockIdx.y * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
#pragma unroll
    for (int r = ty; r < 64; r += 4) {
        const int64_t k = k0 + r, j = j0 + tx;
        tile[r][tx] = k < K && j < R && !(upper && k > j) ? S[k * lds + j] : 0.0;
    }
    __syncthreads();
    oz_slice_tile<D, false>(tile, k0, j0, K, R, nullptr, eexp, nullptr, 0, planes, Ra, r0);
}

// The same for a short K (at most kOzShortK: the coefficients and factors that multiply a
// basis from the right), exponents included, in one launch: a block takes 8 columns over
// all K.  (The column-maximum and slicing kernels and the fill before them took 9 us a
// product at 512 x 64; 5 us now.)
// BAL: row k times the power of two that the left operand's column k was divided by.
constexpr int kOzShortK = 2048;
template <int D, bool BAL>
__global__ void __launch_bounds__(256) oz_slice_cols_short_kernel(int64_t K, int64_t R, const double* __restrict__ S,
                                                                  int64_t lds, int upper,
                                                                  __nv_bfloat16* __restrict__ planes, int64_t Ra,
                                                                  int* __restrict__ eexp, const int* __restrict__ cexp) {
    __shared__ int red[32][9];
    __shared__ int es[8];
    const int64_t j0 = (int64_t)blockIdx.x * 8;
    {
        const int64_t j = j0 + (threadIdx.x & 7);
        int e = kOzZeroExp;
        if (j < R) {
#pragma unroll 4
            for (int64_t k = threadIdx.x >> 3; k < K; k += 32)
                if (!(upper && k > j))
                    e = max(e, BAL ? oz_exp_over(S[k * lds + j], -oz_balance(cexp, k)) : oz_exp(S[k * lds + j]));
        }
        red[threadIdx.x >> 3][threadIdx.x & 7] = e;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        int e = red[0][threadIdx.x];
        for (int y = 1; y < 32; ++y) e = max(e, red[y][threadIdx.x]);
        es[threadIdx.x] = e = oz_norm_exp(e);
        if (j0 + threadIdx.x < R) eexp[j0 + threadIdx.x] = e;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, pr = 2 * (threadIdx.x & 7), sub = (threadIdx.x & 31) >> 3;
    const int units = 2 * (int)(oz_k16(K) / 16);
#pragma unroll 2
    for (int u = warp; u < units; u += 8) {
        const int q = (u & 1) * 4 + sub;
        const int64_t j = j0 + q, k = (int64_t)(u >> 1) * 16 + pr;
        if (j >= R) continue;
        const double x0 = k < K && !(upper && k > j) ? S[k * lds + j] : 0.0;
        const double x1 = k + 1 < K && !(upper && k + 1 > j) ? S[(k + 1) * lds + j] : 0.0;
        const int s0 = BAL && k < K ? oz_balance(cexp, k) : 0, s1 = BAL && k + 1 < K ? oz_balance(cexp, k + 1) : 0;
        oz_store_pair<D>(planes, Ra, j, k, x0, x1, es[q] - s0, es[q] - s1);
    }
}

// ---- the product kernel ------------------------------------------------------
struct OzArgs {
    int64_t M, N, totalg;  // totalg: (row tile, K block) units of one column tile
    int KB, NT, tilen;     // K blocks, column tiles and their width
    int Gg, nslots;        // CTA c: column tile c % NT, unit group c / NT of Gg; partial tiles it may leave
    const int* ea;
    const int* eb;
    double* out;  // C (direct tiles)
    int64_t ldo;
    double alpha, beta;
    int symmetric;
    double* partial;  // [CTA][nslots][128][64]
    int* status;
    long long max_wait;  // limit of one pipeline wait (SM clock cycles)
};

// First unit of group g: the (row tile, K block) units of a column tile are split
// evenly over Gg groups; the NT CTAs of a group (one per column tile) cover the same
// units at the same time, so the A planes they all read come from DRAM once.
__host__ __device__ inline int64_t oz_glo(int g, const OzArgs& a) {
    return (int64_t)g * a.totalg / a.Gg;
}

// (hi + lo 2^-F) 2^(ea + eb - 46), rounded once to nearest even.  In integer arithmetic: a
// warp-wide FP64 instruction takes 16 clocks of the SM's FP64 pipe, and the five that a
// conversion by casts needs bounded the products with a short K (28,000 of 90,000 clocks a
// tile at K = 576).
template <int F>
__device__ inline double oz_value(long long hi, int lo, int ea, int eb) {
    if (ea >= kOzNanExp || eb >= kOzNanExp) return __longlong_as_double(0x7ff8000000000000LL);
    const int E = ea + eb - 46;
    // sign and magnitude: m + r 2^-F
    const long long v = hi + (lo >> F);
    const unsigned r0 = (unsigned)lo & ((1u << F) - 1u);
    const bool neg = v < 0;
    const unsigned r = neg ? ((1u << F) - r0) & ((1u << F) - 1u) : r0;
    const unsigned long long m = neg ? ~(unsigned long long)v + (r0 == 0u ? 1ull : 0ull) : (unsigned long long)v;
    const int lz = __clzll((long long)m), be = 1086 + E - lz;  // biased exponent of the leading bit
    if (m != 0ull && be >= 1 && be <= 2046) {
        // 64 leading bits, the rest ORed into the last one
        unsigned long long w = m << lz;
        w |= lz >= F ? (unsigned long long)r << (lz - F) : (unsigned long long)(r >> (F - lz));
        if (lz < F && (r & ((1u << (F - lz)) - 1u))) w |= 1ull;
        unsigned long long mant = w >> 11;
        mant += ((unsigned)w & 0x7ffu) + ((unsigned)mant & 1u) > 0x400u ? 1ull : 0ull;
        const unsigned long long bits = ((unsigned long long)(be - 1) << 52) + mant;  // a carry raises the exponent
        return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
    }
    // zero, a fraction alone, or a result at the ends of the FP64 range: x 2^E in two steps
    // (the first one is exact)
    const double x = fma((double)lo, F == 8 ? 0x1p-8 : 0x1p-16, (double)hi);
    const int E1 = max(-900, min(E, 1023));
    double y = x * __longlong_as_double((long long)(E1 + 1023) << 52);
    if (E1 != E) y *= __longlong_as_double((long long)(max(-1022, min(E - E1, 1023)) + 1023) << 52);
    return y;
}

// alpha v: no FP64 instruction for 1 and -1
__device__ inline double oz_scale(double alpha, double v) {
    return alpha == 1.0 ? v : (alpha == -1.0 ? -v : alpha * v);
}

// The output rule: out = alpha v + beta out (beta == 0: no read); a symmetric
// product writes each pair (i, j), (j, i) once, from the entry with i <= j.
__device__ inline void oz_store(const OzArgs& a, int64_t i, int64_t j, double v) {
    if (a.symmetric) {
        if (i > j) return;
        a.out[i * a.ldo + j] = v;
        a.out[j * a.ldo + i] = v;
        return;
    }
    double* o = a.out + i * a.ldo + j;
    const double w = oz_scale(a.alpha, v);
    *o = (a.beta != 0.0) ? fma(a.beta, *o, w) : w;
}

// 1.5 2^23: adding it to an integer of magnitude <= 2^22 leaves that integer, plus the
// bits of the constant, in the float's bit pattern (an exact conversion on the FP32 pipe).
constexpr float kOzMagic = 12582912.0f;
constexpr unsigned kOzMagicBits = 0x4B400000u;

// Adds T_g of 8 columns (from column q0 on) to the integer sums.  lo counts units of 2^-40
// with 7 digits (T_6 rounded to it) and of 2^-48 with 8 (T_5 in two parts, T_7 rounded).
template <int N, int D>
__device__ inline void oz_add_slot(int g, int q0, const uint32_t* v, unsigned long long (&hi)[N],
                                   unsigned (&lo)[N]) {
    if (g == 0) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            hi[q0 + q] += (unsigned long long)__float_as_uint(__uint_as_float(v[q]) + kOzMagic) << 32;
    } else if (g <= 4) {
        const int mul = 1 << (32 - 8 * g);  // weight of T_g in hi
#pragma unroll
        for (int q = 0; q < 8; ++q)
            asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hi[q0 + q]) : "r"(__float2int_rn(__uint_as_float(v[q]))), "r"(mul));
    } else if (g == 5) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int t = __float2int_rn(__uint_as_float(v[q]));
            if (D == 7) {
                lo[q0 + q] += (unsigned)t;
            } else {
                hi[q0 + q] += (unsigned long long)(long long)(t >> 8);
                lo[q0 + q] += ((unsigned)t & 255u) << 8;
            }
        }
    } else if (D == 8 && g == 6) {
#pragma unroll
        for (int q = 0; q < 8; ++q) lo[q0 + q] += (unsigned)__float2int_rn(__uint_as_float(v[q]));
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) lo[q0 + q] += __float_as_uint(fmaf(__uint_as_float(v[q]), 0x1p-8f, kOzMagic));
    }
}

// Whether the accumulators of a group start afresh at K block j of a tile.
__device__ inline bool oz_chunk_start(int group, int j) {
    return j == 0 || (group == 0 ? ((j + kOzLowShift) % kOzLowChunk) == 0 : (j % kOzHighChunk) == 0);
}

// The product kernel.  What bounds it: the tensor pipe (28 NC MMA columns of K = 16 a
// stage, 896 clocks at NC = 64) next to L2 (42 KB a stage and CTA).
// Digit plane p of A meets B planes q = 0 .. 6 - p; the products go to the accumulators of
// p + q, which sit side by side in TMEM as the B planes do in shared memory, so that one
// MMA covers several B planes.  The accumulators form two groups, p + q <= 3 (4 MMAs a
// stage) and p + q >= 4 (7 MMAs).  The MMA thread issues kOzRun K blocks for the one, then
// the same K blocks for the other, and the exact-accumulation chunks of the two end at
// different K blocks: while the epilogue reads the accumulators of one group, the MMAs of
// the other run.  With all 7 in one group the tensor pipe stood still at each chunk end.
// Measured, clocks per K block of 16 and CTA (one group, 10 MMAs, before): 10,000^2 x 128
// 1,290 (2,500), 100,000 x 576 times 576 x 64 1,710 (3,100), the projection 576 x 100,000
// times 64 columns 1,700 (2,470; 1,240 would be the DRAM rate of its A planes), width 16
// 1,200 (DRAM-bound).  The MMAs alone take 930; what is left is shared memory, which MMA
// operands and copies share (142 of 128 KB per 1,000 clocks).  Tried and left out: copies
// of A (or B) multicast to a cluster of two CTAs, which changed nothing once the copies
// were long runs, and an L2 prefetch ahead of the copies, which slowed them by a third.
//
// The wide form (D = 8) has 8 digits and accumulators and 36 digit products (12 MMAs and
// 1,152 clocks a K block): 63 bits below a row's (column's) largest entry, where the 7-digit
// form's 55 leave entries 1,000 times smaller than it fewer than FP64's 53.
template <int NC, int D>
__global__ void __launch_bounds__(OzShape<NC, D>::kThreads, 1)
    oz_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, OzArgs a) {
    using S = OzShape<NC, D>;
    constexpr int kSt = S::kStages;
    constexpr int kFrac = D == 7 ? 8 : 16;  // lo counts units of 2^-kFrac of hi's
    extern __shared__ uint8_t dsm[];
    __shared__ __align__(8) uint64_t bars[2 * kSt + 5];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(kSt + s); };
    auto accf = [&](int h) { return bar0 + 8u * (uint32_t)(2 * kSt + h); };      // group h: chunk complete
    auto acce = [&](int h) { return bar0 + 8u * (uint32_t)(2 * kSt + 2 + h); };  // group h: chunk read
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kSt + 4);
    volatile int* abort_flag = &s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x;
    const int nt = c % a.NT, gc = c / a.NT;  // this CTA's column tile and unit group
    const int64_t lo = oz_glo(gc, a), hi = oz_glo(gc + 1, a);
    const int KB = a.KB;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSt; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(accf(h), 1);
            mbar_init(acce(h), S::kEpiWarps);  // one arrival an epilogue warp
        }
        mbar_init(drain, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&s_tmem), S::kTmemCols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        if (elect_one()) {
            // ---- TMA producer: both operands' 7 planes of one 16-wide K block per stage
            bool ok = true;
            int st = 0, issued = 0;
            uint32_t ph = 1;  // parity of the wait for an empty stage (the first round does not wait)
            int mt = (int)(lo / KB), kb = (int)(lo - (int64_t)mt * KB);
            for (int n = (int)(hi - lo); n > 0; --n) {
                if (issued >= kSt) ok = mbar_wait(empty(st), ph, abort_flag, a.max_wait);
                if (!ok) break;
                const uint32_t sA = base + (uint32_t)(st * S::kStage);
                mbar_arrive_expect_tx(full(st), (uint32_t)S::kStage);
                // (coordinates in groups of 16 rows)
                tma_load_3d(sA, &tmA, 0, mt * (kOzM / 16), kb * D, full(st));
                tma_load_3d(sA + S::kStageA, &tmB, 0, nt * (NC / 16), kb * D, full(st));
                if (issued < kSt) ++issued;
                if (++st == kSt) {
                    st = 0;
                    ph ^= 1u;
                }
                if (++kb == KB) {
                    kb = 0;
                    ++mt;
                }
            }
            if (!ok) {
                atomicOr(&a.status[kStTimeout], 1);
                s_abort = 1;
            }
            // before the CTA leaves, every copy issued has landed: the last `issued` stages,
            // oldest first; ph ^ 1 is the parity of the current round
            for (int j = 0; j < issued; ++j) {
                int s = st - issued + j;
                uint32_t fp = ph ^ 1u;
                if (s < 0) {
                    s += kSt;
                    fp ^= 1u;
                }
                mbar_drain(full(s), fp);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            // ---- MMA issuer
            bool ok = true;
            int st = 0;
            uint32_t fph = 0;                // parity of the wait for a full stage
            uint32_t eph[2] = {0, 0};        // parity of the wait for a group that has been read
            bool used[2] = {false, false};
            int kb = (int)(lo % KB);
            for (int left = (int)(hi - lo); left > 0 && ok;) {
                const int nk = min(KB - kb, left);  // K blocks of this tile here
                for (int j0 = 0; j0 < nk && ok; j0 += kOzRun) {
                    const int j1 = min(j0 + kOzRun, nk);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        int s = st;
                        uint32_t f = fph;
                        for (int j = j0; j < j1; ++j) {
                            if (h == 0) {
                                ok = mbar_wait(full(s), f, abort_flag, a.max_wait);
                                if (!ok) break;
                            }
                            const bool start = oz_chunk_start(h, j);
                            if (start) {
                                if (used[h]) {
                                    ok = mbar_wait(acce(h), eph[h], abort_flag, a.max_wait);
                                    if (!ok) break;
                                    eph[h] ^= 1u;
                                }
                                used[h] = true;
                            }
                            fence_after();
                            const uint32_t sA = base + (uint32_t)(s * S::kStage);
                            const uint64_t a0 = sdesc_sw32(sA), b0 = sdesc_sw32(sA + S::kStageA);
                            if (h == 0) {
#pragma unroll
                                for (int p = 0; p < kOzLowSlots; ++p)  // slots p .. 3
                                    mma_bf16(tmem + (uint32_t)(p * NC), a0 + (uint64_t)(p * (kOzPlaneA >> 4)), b0,
                                             idesc_bf16(kOzM, (kOzLowSlots - p) * NC), (start && p == 0) ? 0u : 1u);
                            } else {
#pragma unroll
                                for (int p = 0; p < D; ++p) {  // slots max(4, p) .. D - 1
                                    const int g0 = p < kOzLowSlots ? kOzLowSlots : p;
                                    mma_bf16(tmem + (uint32_t)(g0 * NC), a0 + (uint64_t)(p * (kOzPlaneA >> 4)),
                                             b0 + (uint64_t)((g0 - p) * (S::kPlaneB >> 4)),
                                             idesc_bf16(kOzM, (D - g0) * NC), (start && p == 0) ? 0u : 1u);
                                }
                                commit(empty(s));
                            }
                            if (j + 1 == nk || oz_chunk_start(h, j + 1)) commit(accf(h));
                            if (++s == kSt) {
                                s = 0;
                                f ^= 1u;
                            }
                        }
                        if (!ok) break;
                        if (h == 1) {
                            st = s;
                            fph = f;
                        }
                    }
                }
                left -= nk;
                kb = 0;
            }
            if (!ok) {
                atomicOr(&a.status[kStTimeout], 1);
                s_abort = 1;
            }
            commit(drain);
            mbar_drain(drain, 0);
        }
        __syncwarp();
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, CW of the columns
        constexpr int CW = 4 * NC / S::kEpiWarps;
        const int r = (warp & 3) * 32 + lane, cofs = ((warp - 2) >> 2) * CW;
        const uint32_t t0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cofs;
        uint32_t ph = 0;  // bit h: parity of the wait for group h
        int seg = 0;
        bool ok = true;
        int mt = (int)(lo / KB), kb = (int)(lo - (int64_t)mt * KB);
        for (int left = (int)(hi - lo); left > 0 && ok; ++seg, ++mt) {
            const int nk = min(KB - kb, left);
            // integer sums of the digit products: hi in units of 2^-32 of the leading one
            // (p + q <= 4, exact), lo below them (oz_add_slot), both biased by the magic bits of the chunks added
            unsigned long long hi64[CW];
            unsigned lo32[CW];
#pragma unroll
            for (int q = 0; q < CW; ++q) {
                hi64[q] = 0ull;
                lo32[q] = 0u;
            }
            int nlow = 0, nhigh = 0, nfold = 0;  // chunks added (nfold: since the last carry)
            bool stored = false;
            int jl = min(nk, kOzLowChunk - kOzLowShift), jh = min(nk, kOzHighChunk);  // next chunk ends
            for (bool more = true; more && ok;) {
                const int h = jl <= jh ? 0 : 1;  // the group whose chunk ends next (both at nk: low first)
                int w_ok = 1;
                if (lane == 0) w_ok = mbar_wait(accf(h), (ph >> h) & 1u, abort_flag, a.max_wait) ? 1 : 0;
                w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
                if (!w_ok) {
                    if (lane == 0) {
                        atomicOr(&a.status[kStTimeout], 1);
                        s_abort = 1;
                    }
                    ok = false;
                    break;
                }
                ph ^= 1u << h;
                fence_after();
                // Slot g holds T_g, an integer within 2^24.  8 columns are converted while the
                // next 8 are read; the group goes back to the MMA thread as soon as its last
                // columns are in registers.  T_0 (at most 2^22) and the last T_g, rounded to the
                // unit of lo, convert on the FP32 pipe, the others by F2I.  The loop over slots stays
                // rolled: unrolled, the scheduler gathers so many conversions that the sums
                // no longer fit the 168 registers of a thread.
                const int g1 = h == 0 ? kOzLowSlots : D;
                uint32_t buf[2][8];
                const int g0 = h == 0 ? 0 : kOzLowSlots;
                tmem_ld8_async(t0 + g0 * NC, buf[0]);
                tmem_wait8(buf[0]);
#pragma unroll 1
                for (int g = g0; g < g1; ++g) {
                    const bool lastg = g + 1 == g1;
#pragma unroll
                    for (int q = 0; q < CW; q += 8) {
                        const int b = (q >> 3) & 1;
                        const bool lastq = q + 8 == CW;
                        // (one buffer where 8 columns are all: NC = 16)
                        if (CW > 8 && !(lastq && lastg))
                            tmem_ld8_async(lastq ? t0 + (g + 1) * NC : t0 + g * NC + q + 8, buf[b ^ 1]);
                        if (CW == 8 && lastg) {
                            fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(acce(h));
                        }
                        oz_add_slot<CW, D>(g, q, buf[b], hi64, lo32);
                        if (CW == 8 && !lastg) {
                            tmem_ld8_async(t0 + (g + 1) * NC, buf[0]);
                            tmem_wait8(buf[0]);
                        }
                        if (CW > 8 && !(lastq && lastg)) tmem_wait8(buf[b ^ 1]);
                        if (CW > 8 && q + 16 == CW && lastg) {
                            fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(acce(h));
                        }
                    }
                }
                if (h == 0) {
                    ++nlow;
                    jl = jl == nk ? INT_MAX : min(nk, jl + kOzLowChunk);
                } else {
                    ++nhigh;
                    jh = jh == nk ? INT_MAX : min(nk, jh + kOzHighChunk);
                    if (++nfold == kOzFoldChunks) {
                        nfold = 0;
#pragma unroll
                        for (int q = 0; q < CW; ++q) {  // hi + lo 2^-kFrac unchanged
                            const int t = (int)(lo32[q] - (unsigned)kOzFoldChunks * kOzMagicBits);
                            hi64[q] += (unsigned long long)(long long)(t >> kFrac);
                            lo32[q] = (unsigned)(t & ((1 << kFrac) - 1));
                        }
                    }
                }
                more = jl != INT_MAX || jh != INT_MAX;
                if (more && nhigh < kOzFlushChunks) continue;
                // output: two columns an iteration of a rolled loop that shifts the sums down
                // (their conversion, unrolled over all columns, would not fit the registers)
                const int64_t row = (int64_t)mt * kOzM + r, col0 = (int64_t)nt * NC + cofs;
                const int ea = row < a.M ? a.ea[row] : 0;
                const int eb_lane = lane < CW && col0 + lane < a.N ? a.eb[col0 + lane] : 0;  // column col0 + lane
                const unsigned long long bias = (unsigned long long)((unsigned)nlow * kOzMagicBits) << 32;
                const unsigned lobias = (unsigned)nfold * kOzMagicBits;
                const bool direct = nk == KB && KB <= kOzHighChunk * kOzFlushChunks;
                const bool pair = !direct || (!a.symmetric && (a.ldo & 1) == 0 &&
                                              (reinterpret_cast<uintptr_t>(a.out) & 15) == 0);
                // segments whose tile is cut between CTAs (at most the first and the last one
                // unless the tile is longer than one flush) leave a partial tile
                const int islot = KB <= kOzHighChunk * kOzFlushChunks ? (seg ? 1 : 0) : seg;
                double* o = direct ? a.out + row * a.ldo + col0
                                   : a.partial + (((int64_t)c * a.nslots + islot) * kOzM + r) * kOzN + cofs;
#pragma unroll 1
                for (int cc = 0; cc < CW; cc += 2) {
                    const int eb0 = __shfl_sync(0xffffffffu, eb_lane, cc);
                    const int eb1 = __shfl_sync(0xffffffffu, eb_lane, cc + 1);
                    const int64_t col = col0 + cc;  // columns col, col + 1
                    if (row < a.M && col < a.N) {
                        const bool two = col + 1 < a.N;
                        double2 w = make_double2(0.0, 0.0);
                        w.x = oz_value<kFrac>((long long)(hi64[0] - bias), (int)(lo32[0] - lobias), ea, eb0);
                        if (two) w.y = oz_value<kFrac>((long long)(hi64[1] - bias), (int)(lo32[1] - lobias), ea, eb1);
                        double* oq = o + cc;
                        if (pair && two) {
                            if (direct) {
                                w.x = oz_scale(a.alpha, w.x);
                                w.y = oz_scale(a.alpha, w.y);
                            }
                            if (direct ? a.beta != 0.0 : stored) {
                                const double2 z = *reinterpret_cast<const double2*>(oq);
                                const double beta = direct ? a.beta : 1.0;
                                w.x = fma(beta, z.x, w.x);
                                w.y = fma(beta, z.y, w.y);
                            }
                            *reinterpret_cast<double2*>(oq) = w;
                        } else if (direct) {
                            oz_store(a, row, col, w.x);
                            if (two) oz_store(a, row, col + 1, w.y);
                        } else {
                            *oq = stored ? *oq + w.x : w.x;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < CW; ++q) {
                        hi64[q] = q + 2 < CW ? hi64[q + 2 < CW ? q + 2 : 0] : 0ull;
                        lo32[q] = q + 2 < CW ? lo32[q + 2 < CW ? q + 2 : 0] : 0u;
                    }
                }
                stored = true;
                nlow = nhigh = nfold = 0;
            }
            left -= nk;
            kb = 0;
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, S::kTmemCols);
    }
}

// The tiles whose K range is split over CTAs (or longer than one 64-bit accumulation): row
// tile mt, the nc groups from g0 on, and the slot of group g0's partial tile (the others
// start inside the tile: slot 0).  Listed by the host, as one thread finding them took
// longer than the sums.
struct OzCuts {
    int mt[kOzWave];
    short g0[kOzWave], nc[kOzWave], slot0[kOzWave];
};

// Adds the parts of a cut tile and applies the output rule.  Block (x, y, z): `rows` rows
// from x * rows on of cut y, column tile z.  Few parts: 4 rows at a time, in CTA order.
// Many (a Gram matrix has 152 parts of one tile): a row at a time, four contiguous shares
// of the CTAs, then the shares in order.
__global__ void __launch_bounds__(256) oz_fixup_kernel(OzArgs a, OzCuts cuts, int rows) {
    __shared__ double s_part[4][kOzN];
    const int mt = cuts.mt[blockIdx.y], nc = cuts.nc[blockIdx.y], g0 = cuts.g0[blockIdx.y], nt = blockIdx.z;
    const int cl = threadIdx.x % kOzN, share = threadIdx.x / kOzN;
    const int64_t col = (int64_t)nt * a.tilen + cl;
    const bool in_col = cl < a.tilen && col < a.N;
    const double* first = a.partial + (((int64_t)g0 * a.NT + nt) * a.nslots + cuts.slot0[blockIdx.y]) * kOzM * kOzN;
    const double* rest = a.partial + ((int64_t)g0 * a.NT + nt) * a.nslots * kOzM * kOzN;
    const int64_t step = (int64_t)a.NT * a.nslots * kOzM * kOzN;  // from one group's slot 0 to the next's
    const int r1 = min((int)(blockIdx.x + 1) * rows, (int)min((int64_t)kOzM, a.M - (int64_t)mt * kOzM));
    if (nc < 8) {
#pragma unroll 2
        for (int r = (int)blockIdx.x * rows + share; r < r1; r += 4) {
            const int idx = r * kOzN + cl;
            if (!in_col) continue;
            double acc = first[idx];
            for (int j = 1; j < nc; ++j) acc += rest[j * step + idx];
            oz_store(a, (int64_t)mt * kOzM + r, col, acc);
        }
        return;
    }
    for (int r = (int)blockIdx.x * rows; r < r1; ++r) {
        const int idx = r * kOzN + cl;
        double acc = 0.0;
        if (in_col) {
            int j = nc * share / 4;
            const int j1 = nc * (share + 1) / 4;
            if (j == 0) acc = first[idx], j = 1;
            for (; j + 16 <= j1; j += 16) {  // sixteen loads in flight
                double v[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) v[u] = rest[(j + u) * step + idx];
#pragma unroll
                for (int u = 0; u < 16; ++u) acc += v[u];
            }
#pragma unroll 8
            for (; j < j1; ++j) acc += rest[j * step + idx];
        }
        __syncthreads();
        s_part[share][cl] = acc;
        __syncthreads();
        if (in_col && share == 0)
            oz_store(a, (int64_t)mt * kOzM + r, col, ((acc + s_part[1][cl]) + s_part[2][cl]) + s_part[3][cl]);
    }
}

// ---- host side -------------------------------------------------------------------
struct OzPlan {
    int64_t M, N, K, tiles, totalg;
    int KB, MT, NT, tilen, G, Gg, nslots;
};

// Column tiles of 16, 32 or 64 columns (7 accumulators of 64 fill the tensor memory).
OzPlan oz_plan(int64_t M, int64_t N, int64_t K) {
    OzPlan p{};
    p.M = M;
    p.N = N;
    p.K = K;
    p.tilen = N <= 16 ? 16 : (N <= 32 ? 32 : kOzN);
    p.MT = (int)((M + kOzM - 1) / kOzM);
    p.NT = (int)((N + p.tilen - 1) / p.tilen);
    p.KB = (int)std::max<int64_t>(1, (K + kOzBK - 1) / kOzBK);
    p.tiles = (int64_t)p.MT * p.NT;
    p.totalg = (int64_t)p.MT * p.KB;
    p.Gg = (int)std::max<int64_t>(1, std::min<int64_t>(kOzWave / p.NT, p.totalg));
    p.G = p.Gg * p.NT;
    int maxseg = 1;
    OzArgs a{};
    a.KB = p.KB;
    a.totalg = p.totalg;
    a.Gg = p.Gg;
    for (int g = 0; g < p.Gg; ++g) {
        const int64_t lo = oz_glo(g, a), hi = oz_glo(g + 1, a);
        if (hi > lo) maxseg = std::max<int>(maxseg, (int)((hi - 1) / p.KB - lo / p.KB + 1));
    }
    // partial tiles of a CTA: its first and its last, or all where a tile is longer than
    // one 64-bit accumulation
    p.nslots = p.KB <= kOzHighChunk * kOzFlushChunks ? std::min(maxseg, 2) : maxseg;
    return p;
}

inline size_t oz_planes_bytes(int64_t rows, int64_t K, int dig) {
    return align256((size_t)dig * (size_t)oz_ra(rows) * (size_t)oz_k16(K) * 2);
}

// 3-D tensor map of one operand: dims {16 rows = 256 elements, groups of 16 rows, digits x
// K blocks}, box 512 bytes x box_rows / 16 x digits, copied byte for byte.  Groups past
// `rows` read zeros; the rows past it in the last group hold anything, and only reach output
// rows (columns) that do not exist.
bool make_oz_map(CUtensorMap* map, const void* planes, int64_t rows, int64_t Ra, int64_t K, int box_rows, int dig) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {256, (cuuint64_t)(oz_ra(rows) / 16), (cuuint64_t)(dig * (oz_k16(K) / 16))};
    const cuuint64_t strides[2] = {512, (cuuint64_t)Ra * 32};
    const cuuint32_t box[3] = {256u, (cuuint32_t)(box_rows / 16), (cuuint32_t)dig};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(planes), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
inline size_t oz_partial_bytes(const OzPlan& p) {
    return align256(sizeof(double) * (size_t)p.G * p.nslots * kOzM * kOzN);
}

// One operand of the product kernel: `rows` stored rows of K digits each in the
// K-block-major layout with Ra allocated stored rows, one exponent per stored row.
struct OzView {
    const __nv_bfloat16* planes;
    int64_t rows, K, Ra;
    const int* exps;
};

// cexp: balanced (wide form only).
int oz_slice_rows(tsvd_handle* h, int64_t R, int64_t c0, int64_t c1, const double* S, int64_t lds, bool grow,
                  __nv_bfloat16* planes, int* eexp, cudaStream_t st, const int* cexp = nullptr) {
    if (R == 0) return TSVD_OK;
    // 8 lanes a row; 32 where that leaves fewer warps than the chip has room for
    const bool few = R <= (int64_t)h->sm_count * 32;
    const int64_t rows = few ? 8 : 32;  // of a block
    const int64_t blocks = std::min<int64_t>((R + rows - 1) / rows, (int64_t)h->sm_count * 32);
    const bool wide = h->oz_dig == kOzWideDig;
    const auto kern = grow   ? (few ? oz_slice_rows_kernel<kOzDig, true, 32> : oz_slice_rows_kernel<kOzDig, true, 8>)
                      : cexp ? (few ? oz_slice_rows_kernel<kOzWideDig, false, 32, true>
                                    : oz_slice_rows_kernel<kOzWideDig, false, 8, true>)
                      : wide ? (few ? oz_slice_rows_kernel<kOzWideDig, false, 32>
                                    : oz_slice_rows_kernel<kOzWideDig, false, 8>)
                             : (few ? oz_slice_rows_kernel<kOzDig, false, 32>
                                    : oz_slice_rows_kernel<kOzDig, false, 8>);
    h->launches++;
    kern<<<(unsigned)blocks, 256, 0, st>>>(R, c0, c1, S, lds, planes, oz_ra(R), eexp, cexp);
    TSVD_TRY_CUDA(cudaGetLastError());
    return TSVD_OK;
}

// The column maxima of S alone.
int oz_colmax(tsvd_handle* h, int64_t K, int64_t R, const double* S, int64_t lds, bool upper, int* eexp,
              cudaStream_t st) {
    const unsigned gx = (unsigned)((R + 31) / 32);
    int64_t gy = std::min<int64_t>((K + 255) / 256, std::max<int64_t>(1, (int64_t)h->sm_count * 8 / gx));
    const int64_t rows_per = (K + gy - 1) / gy;
    gy = (K + rows_per - 1) / rows_per;
    h->launches++;
    TSVD_TRY_CUDA(cudaMemsetAsync(eexp, kOzUnset, sizeof(int) * R, st));
    oz_colmax_kernel<<<dim3(gx, (unsigned)std::max<int64_t>(1, gy)), dim3(32, 8), 0, st>>>(K, R, S, lds,
                                                                                           upper ? 1 : 0, rows_per,
                                                                                           eexp);
    TSVD_TRY_CUDA(cudaGetLastError());
    return TSVD_OK;
}

// Ra: allocated stored rows of `planes` (default R); r0: first stored row written; cexp:
// balanced (wide form, K <= kOzShortK).
int oz_slice_cols(tsvd_handle* h, int64_t K, int64_t R, const double* S, int64_t lds, bool upper,
                  __nv_bfloat16* planes, int* eexp, cudaStream_t st, int64_t Ra = -1, int64_t r0 = 0,
                  const int* cexp = nullptr) {
    if (R == 0) return TSVD_OK;
    if (Ra < 0) Ra = oz_ra(R);
    const bool wide = h->oz_dig == kOzWideDig;
    if (K <= kOzShortK && r0 == 0) {
        const auto kern = cexp   ? oz_slice_cols_short_kernel<kOzWideDig, true>
                          : wide ? oz_slice_cols_short_kernel<kOzWideDig, false>
                                 : oz_slice_cols_short_kernel<kOzDig, false>;
        h->launches++;
        kern<<<(unsigned)((R + 7) / 8), 256, 0, st>>>(K, R, S, lds, upper ? 1 : 0, planes, Ra, eexp, cexp);
        TSVD_TRY_CUDA(cudaGetLastError());
        return TSVD_OK;
    }
    TSVD_TRY(oz_colmax(h, K, R, S, lds, upper, eexp, st));
    h->launches++;
    const dim3 sg((unsigned)((oz_k16(K) + 63) / 64), (unsigned)((R + 63) / 64));
    const auto kern = wide ? oz_slice_cols_kernel<kOzWideDig> : oz_slice_cols_kernel<kOzDig>;
    kern<<<sg, 256, 0, st>>>(K, R, S, lds, upper ? 1 : 0, eexp, planes, Ra, r0);
    TSVD_TRY_CUDA(cudaGetLastError());
    return TSVD_OK;
}

template <int NC, int D>
int oz_launch(tsvd_handle* h, int grid, const CUtensorMap& mA, const CUtensorMap& mB, const OzArgs& a,
              cudaStream_t st) {
    using S = OzShape<NC, D>;
    static thread_local int configured = -1;
    if (configured != h->device) {
        TSVD_TRY_CUDA(cudaFuncSetAttribute(oz_gemm_kernel<NC, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           S::kSmem));
        configured = h->device;
    }
    h->launches++;
    oz_gemm_kernel<NC, D><<<grid, S::kThreads, S::kSmem, st>>>(mA, mB, a);
    TSVD_TRY_CUDA(cudaGetLastError());
    return TSVD_OK;
}

int oz_run(tsvd_handle* h, const OzPlan& p, const OzView& va, const OzView& vb, double* partial, double* out,
           int64_t ldo, double alpha, double beta, bool symmetric, int* status, cudaStream_t st) {
    if (p.tiles > 65535) return TSVD_ERR_UNSUPPORTED;
    const int dig = h->oz_dig;
    CUtensorMap mA, mB;
    if (!make_oz_map(&mA, va.planes, p.M, va.Ra, p.K, kOzM, dig)) return TSVD_ERR_CUDA;
    if (!make_oz_map(&mB, vb.planes, p.N, vb.Ra, p.K, p.tilen, dig)) return TSVD_ERR_CUDA;
    OzArgs a{};
    a.M = p.M;
    a.N = p.N;
    a.KB = p.KB;
    a.totalg = p.totalg;
    a.NT = p.NT;
    a.tilen = p.tilen;
    a.Gg = p.Gg;
    a.nslots = p.nslots;
    a.ea = va.exps;
    a.eb = vb.exps;
    a.out = out;
    a.ldo = ldo;
    a.alpha = alpha;
    a.beta = beta;
    a.symmetric = symmetric ? 1 : 0;
    a.partial = partial;
    a.status = status;
    a.max_wait = h->max_wait;
    constexpr int kD = kOzDig, kW = kOzWideDig;
    const auto launch = dig == kW ? (p.tilen == 16 ? oz_launch<16, kW> : (p.tilen == 32 ? oz_launch<32, kW> : oz_launch<64, kW>))
                                  : (p.tilen == 16 ? oz_launch<16, kD> : (p.tilen == 32 ? oz_launch<32, kD> : oz_launch<64, kD>));
    TSVD_TRY(launch(h, p.G, mA, mB, a, st));
    const bool all = p.KB > kOzHighChunk * kOzFlushChunks;
    OzCuts cuts;
    int n = 0;
    auto flush = [&]() -> int {
        if (n == 0) return TSVD_OK;
        h->launches++;
        // a few tiles of many parts: a row a block; many tiles of few parts: 16 rows a block
        const int rows = n * p.NT < 16 ? 1 : 16;
        oz_fixup_kernel<<<dim3((unsigned)(kOzM / rows), (unsigned)n, (unsigned)p.NT), 256, 0, st>>>(a, cuts, rows);
        n = 0;
        TSVD_TRY_CUDA(cudaGetLastError());
        return TSVD_OK;
    };
    auto add = [&](int mt, int g0) -> int {  // row tile mt, first held by group g0
        int nc = 1;
        while (g0 + nc < p.Gg && oz_glo(g0 + nc, a) < (int64_t)(mt + 1) * p.KB) ++nc;
        const int first = (int)(oz_glo(g0, a) / p.KB);
        cuts.mt[n] = mt;
        cuts.g0[n] = (short)g0;
        cuts.nc[n] = (short)nc;
        cuts.slot0[n] = (short)(all ? mt - first : (mt > first ? 1 : 0));
        return ++n == kOzWave ? flush() : TSVD_OK;
    };
    if (all) {
        for (int mt = 0, g = 0; mt < p.MT; ++mt) {
            while (g + 1 < p.Gg && oz_glo(g + 1, a) <= (int64_t)mt * p.KB) ++g;
            TSVD_TRY(add(mt, g));
        }
    } else {
        int done = -1;  // row tiles that a group starts inside, each once
        for (int g = 1; g < p.Gg; ++g) {
            const int64_t u = oz_glo(g, a);
            const int mt = (int)(u / p.KB);
            if (mt == done || u == (int64_t)mt * p.KB) continue;
            done = mt;
            TSVD_TRY(add(mt, g - 1));
        }
    }
    TSVD_TRY(flush());
    return TSVD_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
bool oz_worth(int64_t M, int64_t N, int64_t K) {
    // below ~30 MFLOP the FP64 pipe finishes before the slicing passes would
    const int64_t tiles = ((M + kOzM - 1) / kOzM) * ((N + kOzN - 1) / kOzN);
    return M > 0 && N > 0 && K >= 32 && tiles <= 65535 && N <= 65535 * 32 && 2.0 * (double)M * N * K >= 3.0e7;
}

size_t oz_ws_bound(int64_t qmax, int64_t smax, int64_t bmax, int dig) {
    // planes and exponents of the largest operands of either product, and split-K
    // partial tiles for at most (tiles + 2 per CTA of one wave) tiles
    const size_t tn = oz_planes_bytes(smax, qmax, dig) + oz_planes_bytes(bmax, qmax, dig);
    const size_t nn = oz_planes_bytes(qmax, smax, dig) + oz_planes_bytes(bmax, smax, dig);
    const size_t ex = align256(sizeof(int) * (size_t)(qmax + smax)) + align256(sizeof(int) * (size_t)(smax + bmax));
    const int64_t tiles = ((smax + kOzM - 1) / kOzM) * ((bmax + kOzN - 1) / kOzN);
    const size_t part = align256(sizeof(double) * (size_t)(tiles + 2 * kOzWave) * kOzM * kOzN);
    return std::max(tn, nn) + ex + part + 4096;
}

size_t oz_standalone_ws(int64_t q, int64_t s, int b, bool keep) {
    constexpr int kW = kOzWideDig;
    size_t bytes = oz_ws_bound(q, keep ? b : std::max<int64_t>(s, b), b, kW);
    if (s > 0 && keep) {
        bytes += oz_cache_bytes(q, s, true, kW) + oz_cache_bytes(q, s, false, kW);
        bytes += std::max(oz_tn_ws(q, s, b, false, true, kW), oz_nn_ws(q, s, b, true, kW));
    }
    // worth it only if one of the products is
    const bool worth = oz_worth(b, b, q) || oz_worth(q, b, b) || (s > 0 && (oz_worth(s, b, q) || oz_worth(q, b, s)));
    return worth && bytes <= kOzStandaloneMax ? bytes : 0;
}

namespace {

OzView view_of(const __nv_bfloat16* planes, int64_t rows, int64_t K, const int* exps) {
    return OzView{planes, rows, K, oz_ra(rows), exps};
}

// The cached planes of columns [0, s) (cols layout: stored rows) or of the first s
// columns of every row (rows layout: K = s).
OzView view_of_cache(const OzCache& c, int64_t s) {
    return c.cols_layout ? OzView{c.planes, s, c.rows, oz_ra(c.cols), c.exps}
                         : OzView{c.planes, c.rows, s, oz_ra(c.rows), c.exps};
}

}  // namespace

size_t oz_tn_ws(int64_t q, int64_t s, int64_t b, bool symmetric, bool cached_x, int dig) {
    const OzPlan p = oz_plan(s, b, q);
    Arena ar;
    if (!cached_x) {
        ar.take<char>(oz_planes_bytes(p.M, p.K, dig));
        ar.take<int>((size_t)p.M);
    }
    if (!symmetric || cached_x) {
        ar.take<char>(oz_planes_bytes(p.N, p.K, dig));
        ar.take<int>((size_t)p.N);
    }
    ar.take<char>(oz_partial_bytes(p));
    return ar.off;
}

size_t oz_nn_ws(int64_t q, int64_t s, int64_t b, bool cached_x, int dig) {
    const OzPlan p = oz_plan(q, b, s);
    Arena ar;
    if (!cached_x) {
        ar.take<char>(oz_planes_bytes(p.M, p.K, dig));
        ar.take<int>((size_t)p.M);
    }
    ar.take<char>(oz_planes_bytes(p.N, p.K, dig));
    ar.take<int>((size_t)p.N);
    if (dig == kOzWideDig && !cached_x) ar.take<int>((size_t)p.K);
    ar.take<char>(oz_partial_bytes(p));
    return ar.off;
}

size_t oz_a_ws(int64_t M, int64_t N, int64_t w) {
    return std::max(oz_nn_ws(M, N, w, true), oz_tn_ws(M, N, w, false, true));
}

int oz_gemm_tn(tsvd_handle* h, int64_t q, int64_t s, int64_t b, const double* X, int64_t ldx, const double* Z,
               int64_t ldz, double* C, int64_t ldc, bool symmetric, void* ws, size_t ws_bytes, int* status,
               cudaStream_t st, const OzCache* xc) {
    const OzPlan p = oz_plan(s, b, q);
    Arena ar{static_cast<char*>(ws), ws_bytes, 0};
    OzView va{}, vb{};
    if (xc) {
        va = view_of_cache(*xc, s);
    } else {
        __nv_bfloat16* pa = reinterpret_cast<__nv_bfloat16*>(ar.take<char>(oz_planes_bytes(p.M, p.K, h->oz_dig)));
        int* ea = ar.take<int>((size_t)p.M);
        if (!ar.fits()) return TSVD_ERR_WORKSPACE;
        TSVD_TRY(oz_slice_cols(h, q, s, X, ldx, false, pa, ea, st));
        va = view_of(pa, s, q, ea);
    }
    if (symmetric && !xc) {
        vb = va;
    } else {
        __nv_bfloat16* pb = reinterpret_cast<__nv_bfloat16*>(ar.take<char>(oz_planes_bytes(p.N, p.K, h->oz_dig)));
        int* eb = ar.take<int>((size_t)p.N);
        if (!ar.fits()) return TSVD_ERR_WORKSPACE;
        TSVD_TRY(oz_slice_cols(h, q, b, Z, ldz, false, pb, eb, st));
        vb = view_of(pb, b, q, eb);
    }
    const size_t pbytes = oz_partial_bytes(p);
    double* part = pbytes ? reinterpret_cast<double*>(ar.take<char>(pbytes)) : nullptr;
    if (!ar.fits()) return TSVD_ERR_WORKSPACE;
    return oz_run(h, p, va, vb, part, C, ldc, 1.0, 0.0, symmetric, status, st);
}

int oz_gemm_nn(tsvd_handle* h, int64_t q, int64_t s, int64_t b, double alpha, const double* X, int64_t ldx,
               const double* Mm, int64_t ldm, double beta, double* Y, int64_t ldy, bool upper, void* ws,
               size_t ws_bytes, int* status, cudaStream_t st, const OzCache* xc) {
    const OzPlan p = oz_plan(q, b, s);
    Arena ar{static_cast<char*>(ws), ws_bytes, 0};
    OzView va{};
    // Wide form, triangular M (the normalisation Y L^-T of a block whose columns may differ by
    // orders of magnitude): balanced by the columns of X, so that one exponent a row serves all
    // of them.  Error of Q against 1e-28 arithmetic, 87,413 x 128 with columns from 1 to 1e-3:
    // 4.6e-16 without, 1.1e-16 on the FP64 pipe.
    const bool bal = h->oz_dig == kOzWideDig && upper && !xc && s <= kOzShortK;
    int* cexp = nullptr;
    if (xc) {
        va = view_of_cache(*xc, s);
    } else {
        __nv_bfloat16* pa = reinterpret_cast<__nv_bfloat16*>(ar.take<char>(oz_planes_bytes(p.M, p.K, h->oz_dig)));
        int* ea = ar.take<int>((size_t)p.M);
        if (h->oz_dig == kOzWideDig) cexp = ar.take<int>((size_t)p.K);
        if (!ar.fits()) return TSVD_ERR_WORKSPACE;
        if (!bal) cexp = nullptr;
        if (bal) TSVD_TRY(oz_colmax(h, q, s, X, ldx, false, cexp, st));
        TSVD_TRY(oz_slice_rows(h, q, 0, s, X, ldx, false, pa, ea, st, cexp));
        va = view_of(pa, q, s, ea);
    }
    __nv_bfloat16* pb = reinterpret_cast<__nv_bfloat16*>(ar.take<char>(oz_planes_bytes(p.N, p.K, h->oz_dig)));
    int* eb = ar.take<int>((size_t)p.N);
    const size_t pbytes = oz_partial_bytes(p);
    double* part = pbytes ? reinterpret_cast<double*>(ar.take<char>(pbytes)) : nullptr;
    if (!ar.fits()) return TSVD_ERR_WORKSPACE;
    TSVD_TRY(oz_slice_cols(h, s, b, Mm, ldm, upper, pb, eb, st, -1, 0, cexp));
    return oz_run(h, p, va, view_of(pb, b, s, eb), part, Y, ldy, alpha, beta, false, status, st);
}

// ---- caches of operands that many products read ----------------------------------
size_t oz_cache_bytes(int64_t rows, int64_t cols, bool cols_layout, int dig) {
    Arena ar;
    OzCache c;
    oz_cache_carve(c, ar, nullptr, 0, rows, cols, cols_layout, false, dig);
    return ar.off;
}

void oz_cache_carve(OzCache& c, Arena& ar, const double* src, int64_t ld, int64_t rows, int64_t cols,
                    bool cols_layout, bool grows, int dig) {
    c = OzCache{};
    c.src = src;
    c.ld = ld;
    c.rows = rows;
    c.cols = cols;
    c.cols_layout = cols_layout;
    c.grows = grows;
    const int64_t srows = cols_layout ? cols : rows, K = cols_layout ? rows : cols;
    c.planes = reinterpret_cast<__nv_bfloat16*>(ar.take<char>(oz_planes_bytes(srows, K, dig)));
    c.exps = ar.take<int>((size_t)srows);
    c.valid = 0;
}

int oz_cache_slice(tsvd_handle* h, OzCache& c, int64_t c0, int64_t c1, cudaStream_t st) {
    if (c0 > c.valid || c1 > c.cols || c0 > c1) return TSVD_ERR_INVALID_ARG;
    if (c1 > c0) {
        if (c.cols_layout) {
            // stored rows [c0, c1): the columns' own exponents
            TSVD_TRY(oz_slice_cols(h, c.rows, c1 - c0, c.src + c0, c.ld, false, c.planes, c.exps + c0, st,
                                   oz_ra(c.cols),
                                   c0));
        } else {
            // per-row exponents of a matrix that does not grow need the whole rows at once
            if (!c.grows && (c0 != 0 || c1 != c.cols)) return TSVD_ERR_INVALID_ARG;
            TSVD_TRY(oz_slice_rows(h, c.rows, c0, c1, c.src, c.ld, c.grows, c.planes, c.exps, st));
        }
    }
    c.valid = c1;
    return TSVD_OK;
}

int oz_cache_slice_both(tsvd_handle* h, OzCache& rows, OzCache& cols, cudaStream_t st) {
    const int64_t M = rows.rows, N = rows.cols;
    if (rows.cols_layout || rows.grows || !cols.cols_layout || cols.src != rows.src || cols.ld != rows.ld ||
        cols.rows != M || cols.cols != N)
        return TSVD_ERR_INVALID_ARG;
    const int64_t gy = (M + 127) / 128, ty = (std::max(M, oz_k16(M)) + 63) / 64;
    if (gy > 65535 || ty > 65535) {  // (grid limit) one layout at a time
        TSVD_TRY(oz_cache_slice(h, rows, 0, N, st));
        return oz_cache_slice(h, cols, 0, N, st);
    }
    TSVD_TRY_CUDA(cudaMemsetAsync(rows.exps, kOzUnset, sizeof(int) * M, st));
    TSVD_TRY_CUDA(cudaMemsetAsync(cols.exps, kOzUnset, sizeof(int) * N, st));
    h->launches += 2;
    oz_max_both_kernel<<<dim3((unsigned)((N + 255) / 256), (unsigned)gy), 256, 0, st>>>(M, N, rows.src, rows.ld,
                                                                                       rows.exps, cols.exps);
    const auto kern = h->oz_dig == kOzWideDig ? oz_slice_both_kernel<kOzWideDig> : oz_slice_both_kernel<kOzDig>;
    kern<<<dim3((unsigned)((oz_k16(N) + 63) / 64), (unsigned)ty), 256, 0, st>>>(
        M, N, rows.src, rows.ld, rows.exps, cols.exps, rows.planes, oz_ra(M), cols.planes, oz_ra(N));
    TSVD_TRY_CUDA(cudaGetLastError());
    rows.valid = cols.valid = N;
    return TSVD_OK;
}

int oz_cache_truncate(tsvd_handle* h, OzCache& c, int64_t v, cudaStream_t st) {
    if (v >= c.valid) return TSVD_OK;
    c.valid = 0;
    // Rows layout: a row's exponent may stem from the columns dropped here (a block that
    // was not orthonormal, or not finite), and a product of the first v columns reads the
    // whole last K block: the rest is sliced again.
    if (!c.cols_layout && v > 0) return oz_cache_slice(h, c, 0, v, st);
    c.valid = v < 0 ? 0 : v;
    return TSVD_OK;
}

const OzCache* oz_find_cache(const tsvd_handle* h, const double* X, int64_t ldx, int64_t rows, int64_t s,
                             bool cols_layout) {
    for (const OzCache* c : h->oz_caches)
        if (c && c->src == X && c->ld == ldx && c->rows == rows && c->cols_layout == cols_layout && s <= c->valid &&
            // rows layout: the product reads whole 16-wide K blocks, zero past `valid` only
            (cols_layout || s == c->valid || s % 16 == 0))
            return c;
    return nullptr;
}

}  // namespace tsvd
