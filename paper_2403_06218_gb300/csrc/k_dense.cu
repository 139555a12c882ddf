// Dense FP64 kernels of the orthogonalisation building blocks (Table 1):
//   gemm_tn   C = X^T Z        Gram W = Q^T Q (Alg. 4 S1/S4, Alg. 5 S3/S8),
//                              projection H = P^T Q (Alg. 5 S1/S6), A^T X for dense A;
//   gemm_nn   Y = b Y + a X M  update Q - P H (Alg. 5 S2/S7), TRSM applied as the
//                              product with L^{-T} (Alg. 4 S3/S6, Alg. 5 S5/S10),
//                              Ritz/restart products (Alg. 1 S6/S7, Alg. 2 S7-S9), A X;
//   chol_inv  W = L L^T and L^{-T} of the b x b Gram matrix (POTRF of Table 1; one
//             CTA, or a cluster of 8 CTAs for b >= 64);
//   trmm      R = Lbar^T L^T (Alg. 4 S7, Alg. 5 S11);
// plus the Philox/Box-Muller start block, residual column norms, the Lanczos
// residual estimate and the output sign convention.
//
// On GB300 the FP64 pipe issues 2 DFMA/clk/SM (about 1.2 TFLOP/s for the chip),
// which puts every one of these products far above the FP64 ridge point: the
// design goal is the minimum number of DFMAs spread over all SMs, not memory
// traffic.  Symmetric Gram matrices compute only their upper half, triangular
// factors skip their zero half at warp granularity, and split-K partial sums
// are reduced in a fixed order so results are bitwise reproducible.
#include <cooperative_groups.h>

#include <algorithm>

#include "fp64_rsqrt.cuh"
#include "tsvd_internal.cuh"

namespace tsvd {
namespace {

// ---------------------------------------------------------------------------
// gemm_tn: CTA = 4 warps computes a 32 x 32 region of C over one row slab.
// Warp (wr, wc) owns a 16 x 16 sub-tile; lane owns C[i][jg .. jg+7].
// ---------------------------------------------------------------------------
constexpr int kTnR = 32;
constexpr int kTnKc = 32;

__device__ inline void decode_upper(int lin, int nr, int& ri, int& rj) {
    int r = 0;
    while (lin >= nr - r) {
        lin -= nr - r;
        ++r;
    }
    ri = r;
    rj = r + lin;
}

// TI: input element type (also the accumulation type within a slab); TW: type written.
template <typename TI, typename TW>
__global__ void __launch_bounds__(128, 7) gemm_tn_kernel(int64_t q, int64_t s, int64_t b,
                                                      const TI* __restrict__ X, int64_t ldx,
                                                      const TI* __restrict__ Z, int64_t ldz,
                                                      TW* __restrict__ out, int64_t ldo,
                                                      int64_t slab_stride, int64_t slab_rows, int symmetric,
                                                      int nreg_s, int nreg_b) {
    __shared__ TI Xs[kTnKc][kTnR];
    __shared__ TI Zs[kTnKc][kTnR];
    int ri, rj;
    if (symmetric) {
        decode_upper((int)blockIdx.x, nreg_s, ri, rj);
    } else {
        ri = (int)blockIdx.x / nreg_b;
        rj = (int)blockIdx.x % nreg_b;
    }
    const int64_t r0 = (int64_t)blockIdx.y * slab_rows;
    const int64_t r1 = min(q, r0 + slab_rows);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wr = warp >> 1, wc = warp & 1;
    const int i = lane >> 1, jg = (lane & 1) * 8;
    // (a sub-tile below the diagonal or wholly past the last row or column has no work)
    const bool active = !(symmetric && ri == rj && wr > wc) && (int64_t)ri * kTnR + wr * 16 < s &&
                        (int64_t)rj * kTnR + wc * 16 < b;
    TI acc[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = TI(0);
    const int64_t xc0 = (int64_t)ri * kTnR, zc0 = (int64_t)rj * kTnR;
    for (int64_t k0 = r0; k0 < r1; k0 += kTnKc) {
        for (int idx = tid; idx < kTnKc * kTnR; idx += 128) {
            const int rr = idx / kTnR, cc = idx % kTnR;
            const int64_t row = k0 + rr;
            const bool rin = row < r1;
            Xs[rr][cc] = (rin && xc0 + cc < s) ? X[row * ldx + xc0 + cc] : TI(0);
            Zs[rr][cc] = (rin && zc0 + cc < b) ? Z[row * ldz + zc0 + cc] : TI(0);
        }
        __syncthreads();
        if (active) {
            const int kn = (int)min((int64_t)kTnKc, r1 - k0);
#pragma unroll 4
            for (int kk = 0; kk < kn; ++kk) {
                const TI x = Xs[kk][wr * 16 + i];
                const TI* zr = &Zs[kk][wc * 16 + jg];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[t] = fma(x, zr[t], acc[t]);
            }
        }
        __syncthreads();
    }
    if (!active) return;
    const int64_t orow = xc0 + wr * 16 + i;
    if (orow >= s) return;
    TW* o = out + (int64_t)blockIdx.y * slab_stride + orow * ldo + zc0 + wc * 16 + jg;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        if (zc0 + wc * 16 + jg + t < b) o[t] = (TW)acc[t];
    }
}

// C[i][j] = sum over slabs of partial[slab][i][j] in a fixed order: thread
// (x, y) of a 32 x 8 block sums slabs y, y + 8, ... of element x, then the 8
// partial sums are added in y order.  Symmetric reads the upper element for both
// halves.
template <typename TC>
__global__ void __launch_bounds__(256) gemm_tn_reduce_kernel(int64_t s, int64_t b, int slabs,
                                                             const double* __restrict__ partial, int64_t slab_stride,
                                                             TC* __restrict__ C, int64_t ldc, int symmetric) {
    __shared__ double red[8][33];
    const int64_t idx = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const bool in = idx < s * b;
    int64_t i = 0, j = 0, src = 0;
    if (in) {
        i = idx / b;
        j = idx % b;
        const int64_t ii = (symmetric && i > j) ? j : i;
        const int64_t jj = (symmetric && i > j) ? i : j;
        src = ii * b + jj;
    }
    double acc = 0.0;
    if (in)
        for (int sl = threadIdx.y; sl < slabs; sl += 8) acc += partial[(int64_t)sl * slab_stride + src];
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && in) {
        double t = red[0][threadIdx.x];
#pragma unroll
        for (int y = 1; y < 8; ++y) t += red[y][threadIdx.x];
        C[i * ldc + j] = (TC)t;
    }
}

struct TnPlan {
    int nreg_s, nreg_b, regions, slabs;
    int64_t slab_rows;
};

// One full wave of the kernel on a 152-SM GB300: 7 resident CTAs per SM for the
// FP64 kernel (its 72 registers x 128 threads and 16 KB of shared memory allow 7),
// 16 for the 64-thread FP32 kernel (bounded to 64 registers, which it fits without
// spilling).  Splitting K so that regions x slabs fills
// exactly one wave keeps every SM equally busy; a fixed target (rather than the
// device's SM count) keeps the split, the workspace size and the summation order
// independent of the device.
constexpr int64_t kTnWave = 152 * 7;
constexpr int64_t kTnWaveF32 = 152 * 16;

// More slabs (of 16 rows and up) for a product that would leave half the SMs without a CTA:
// its time is that of one CTA's rows, 32 x 32 x 32 FP64 steps taking 8 us of an SM
// (512 x 64 by 512 x 16: 107 us in 2 slabs of 256 rows).  Only while the partial sums stay
// within kTnExtra bytes, which every FP64 workspace has room for.
constexpr size_t kTnExtra = 1 << 20;

TnPlan tn_plan(int64_t q, int64_t s, int64_t b, bool symmetric, int elem_bytes, bool extra) {
    TnPlan p;
    p.nreg_s = (int)((s + kTnR - 1) / kTnR);
    p.nreg_b = (int)((b + kTnR - 1) / kTnR);
    p.regions = symmetric ? p.nreg_s * (p.nreg_s + 1) / 2 : p.nreg_s * p.nreg_b;
    int64_t slabs = (elem_bytes == 4 ? kTnWaveF32 : kTnWave) / p.regions;
    const int64_t max_slabs = (q + 255) / 256;
    if (slabs > max_slabs) slabs = max_slabs;
    if (slabs > 65535) slabs = 65535;
    if (slabs < 1) slabs = 1;
    int64_t align = kTnKc;
    if (extra && elem_bytes == 8 && p.regions * slabs < 76) {
        const int64_t fit = (int64_t)(kTnExtra / sizeof(double)) / (s * b);
        const int64_t more = std::min<int64_t>(std::min<int64_t>((q + 15) / 16, (152 + p.regions - 1) / p.regions), fit);
        if (more > slabs) {
            slabs = more;
            align = 16;
        }
    }
    int64_t rows = (q + slabs - 1) / slabs;
    rows = (rows + align - 1) / align * align;
    if (rows < align) rows = align;
    p.slab_rows = rows;
    p.slabs = (int)((q + rows - 1) / rows);
    if (p.slabs < 1) p.slabs = 1;
    return p;
}

// ---------------------------------------------------------------------------
// gemm_nn: CTA = 4 warps, 32 rows; lane = row, warp w owns CW columns of the
// current panel (4*CW columns); CTAs (x, y), (x, y + gridDim.y) ... of a row of the grid
// share the panels.  X tile and M chunk staged in shared memory,
// output staged for coalesced stores.
// ---------------------------------------------------------------------------
// Accumulation in TX (the precision of the tall operand); M is converted to TX on load.
template <int CW, typename TX, typename TM, typename TY>
__global__ void __launch_bounds__(128) gemm_nn_kernel(int64_t q, int64_t s, int64_t b, double alpha,
                                                      const TX* __restrict__ X, int64_t ldx,
                                                      const TM* __restrict__ M, int64_t ldm, double beta,
                                                      TY* Y, int64_t ldy, int upper) {
    constexpr int PW = 4 * CW;
    __shared__ TX Xs[32][33];
    __shared__ TX Ms[32][PW + 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    for (int64_t c0 = (int64_t)blockIdx.y * PW; c0 < b; c0 += (int64_t)gridDim.y * PW) {
        TX acc[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = TX(0);
        const int64_t jw_hi = c0 + (int64_t)(warp + 1) * CW - 1;  // last column of this warp
        int64_t kmax = s;
        if (upper) kmax = min(s, c0 + PW);
        for (int64_t k0 = 0; k0 < kmax; k0 += 32) {
            for (int idx = tid; idx < 32 * 32; idx += 128) {
                const int rr = idx >> 5, kk = idx & 31;
                const int64_t row = r0 + rr, k = k0 + kk;
                Xs[rr][kk] = (row < q && k < s) ? X[row * ldx + k] : TX(0);
            }
            for (int idx = tid; idx < 32 * PW; idx += 128) {
                const int kk = idx / PW, cc = idx % PW;
                const int64_t k = k0 + kk, col = c0 + cc;
                const bool in = k < s && col < b && !(upper && k > col);
                Ms[kk][cc] = in ? (TX)M[k * ldm + col] : TX(0);
            }
            __syncthreads();
            if (!(upper && k0 > jw_hi) && c0 + warp * CW < b) {
                const int kn = (int)min((int64_t)32, kmax - k0);
#pragma unroll 4
                for (int kk = 0; kk < kn; ++kk) {
                    const TX x = Xs[lane][kk];
                    const TX* mr = &Ms[kk][warp * CW];
#pragma unroll
                    for (int c = 0; c < CW; ++c) acc[c] = fma(x, mr[c], acc[c]);
                }
            }
            __syncthreads();
        }
        // stage through shared memory (reusing Ms) for coalesced stores
#pragma unroll
        for (int c = 0; c < CW; ++c) Ms[lane][warp * CW + c] = acc[c];
        __syncthreads();
        for (int idx = tid; idx < 32 * PW; idx += 128) {
            const int rr = idx / PW, cc = idx % PW;
            const int64_t row = r0 + rr, col = c0 + cc;
            if (row < q && col < b) {
                TY* y = Y + row * ldy + col;
                const TX v = (TX)alpha * Ms[rr][cc];
                *y = (beta != 0.0) ? (TY)fma((TX)beta, (TX)*y, v) : (TY)v;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// chol_inv: one CTA of 256 threads.  Right-looking Cholesky of the lower triangle
// in shared memory (breakdown test d <= b*eps*max_i W_ii), then L^{-1} by
// right-looking forward substitution, stored transposed in the upper triangle of
// the same array (row k of L^{-1} is final once scaled; the rows below it take
// a rank-1 update).  GB300's FP64 pipe costs a warp instruction 16 cycles
// whatever its active lanes, so every FP64 phase is a flat loop over whole
// warps of independent elements (no per-thread chains of varying length), and
// the one scalar step per column (1/sqrt of the pivot) is an FP32 estimate with
// two FP64 Newton steps.
// ---------------------------------------------------------------------------
__device__ inline void tri_decode(int idx, int& ii, int& kk) {
    int r = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
    while (r * (r + 1) / 2 > idx) --r;
    while ((r + 1) * (r + 2) / 2 <= idx) ++r;
    ii = r;
    kk = idx - r * (r + 1) / 2;
}

__global__ void __launch_bounds__(256) chol_inv_kernel(int b, const double* __restrict__ W, double* __restrict__ Lt,
                                                       double* __restrict__ Mt, int* status) {
    extern __shared__ double sm[];
    const int ld = b + 1;
    double* A = sm;                    // lower: L; upper (transposed): L^{-1}
    double* dinv = sm + (size_t)b * ld; // 1 / L_jj
    __shared__ double s_thresh;
    __shared__ int s_bad;
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int idx = tid; idx < b * b; idx += nt) {
        const int i = idx / b, j = idx % b;
        A[i * ld + j] = (j <= i) ? W[idx] : 0.0;  // the upper part starts as zero (L^{-1} = I - ...)
    }
    __syncthreads();
    if (tid == 0) {
        double wmax = 0.0;
        int bad = 0;
        for (int i = 0; i < b; ++i) {
            const double d = A[i * ld + i];
            if (!isfinite(d)) bad = 2;
            if (d > wmax) wmax = d;
        }
        if (bad == 0 && !(wmax > 0.0)) bad = 1;
        s_bad = bad;
        s_thresh = (double)b * kEps * wmax;
    }
    __syncthreads();
    for (int j = 0; j < b && s_bad == 0; ++j) {
        if (tid == 0) {
            const double d = A[j * ld + j];
            if (!isfinite(d) || !(d > s_thresh)) {
                s_bad = isfinite(d) ? 1 : 2;
            } else {
                const double y = rsqrt_fp64(d);
                A[j * ld + j] = d * y;  // L_jj
                dinv[j] = y;
            }
        }
        __syncthreads();
        if (s_bad) break;
        const double inv = dinv[j];
        for (int i = j + 1 + tid; i < b; i += nt) A[i * ld + j] *= inv;
        __syncthreads();
        const int nn = b - j - 1;
        const int cnt = nn * (nn + 1) / 2;
        for (int idx = tid; idx < cnt; idx += nt) {
            int ii, kk;
            tri_decode(idx, ii, kk);
            const int i = j + 1 + ii, k = j + 1 + kk;
            A[i * ld + k] = fma(-A[i * ld + j], A[k * ld + j], A[i * ld + k]);
        }
        __syncthreads();
    }
    if (s_bad) {
        if (tid == 0) atomicOr(&status[s_bad == 2 ? kStNonfinite : kStBreakdown], 1);
        for (int idx = tid; idx < b * b; idx += nt) {
            const double v = (idx / b == idx % b) ? 1.0 : 0.0;
            Lt[idx] = v;
            Mt[idx] = v;
        }
        return;
    }
    // X = L^{-1}: for k = 0..b-1, row k of X (columns c <= k) is scaled by 1/L_kk and
    // is then final; rows i > k take X[i][c] -= L[i][k] X[k][c].  X[i][c] (c < i) is
    // held at A[c][i]; the diagonal of X is dinv.
    for (int k = 0; k < b; ++k) {
        const double ik = dinv[k];
        for (int c = tid; c < k; c += nt) A[c * ld + k] *= ik;
        __syncthreads();
        const int rows = b - k - 1, cols = k + 1;
        for (int idx = tid; idx < rows * cols; idx += nt) {
            const int i = k + 1 + idx / cols, c = idx % cols;
            const double xkc = (c == k) ? ik : A[c * ld + k];
            A[c * ld + i] = fma(-A[i * ld + k], xkc, A[c * ld + i]);
        }
        __syncthreads();
    }
    // Lt = L^T and Mt = L^{-T} = X^T, both upper
    for (int idx = tid; idx < b * b; idx += nt) {
        const int i = idx / b, j = idx % b;
        Lt[idx] = (j >= i) ? A[j * ld + i] : 0.0;
        Mt[idx] = (j > i) ? A[i * ld + j] : (j == i ? dinv[i] : 0.0);
    }
}

// ---------------------------------------------------------------------------
// chol_inv on a cluster of kCholCluster CTAs (b >= kCholClusterMin): forward elimination of
// [A | I], which leaves L^T's columns and M = L^{-1}, with the FP64 work spread over 8 SMs (one
// SM's FP64 pipe, 2 DFMA/clk, bounds the one-CTA kernel above).  Row i belongs to CTA i mod 8,
// column c of M's panel rows to CTA c mod 8.  Per panel of 16 columns:
//   1. warps 0-3 of every CTA factor the 16 x 16 diagonal block, lanes 0-15 a row each and warp w
//      columns w, w + 4, ... (the same numbers and code in every CTA, so every CTA takes the same
//      breakdown decision), while lanes 16-31 take its own 16 rows below through the same steps,
//      which is their substitution L[i][P] = A[i][P] L11^{-T}.  One CTA barrier a pivot; the next
//      pivot's warp updates that column before its others;
//   2. a step behind, warps 4-7 substitute the own columns of the panel's rows of M, a column a
//      lane and rows w, w + 4, ... a warp;
//   3. both go to every CTA (distributed shared memory); cluster barrier;
//   4. rank-16 update of the own rows below, A[i][k] -= L[i][P] L[k][P]^T and M[i][c] -=
//      L[i][P] M[P][c], 16 threads a row; the next panel's rows go out: its diagonal block to
//      every CTA, its rows of M to their columns' owners; cluster barrier.
// Bound by the chain of the pivots (16 steps of 1/sqrt, scale, update a panel) and, at b = 128,
// by the FP64 pipe in the updates.  One warp has a quarter of the SM's FP64 pipe (64 clocks an
// instruction), hence the four warps: b = 128 takes 133 us and b = 64 56 us; with steps 1 and 2 in
// a warp each they took 218 us and 100 us (1,700 clocks a pivot); before, with the pivot steps through shared memory, a
// chain of 136 dependent FMAs a row for its substitution and the inverse in a pass of its own,
// 296 us and 131 us.
// The updates sum 16 products per panel before subtracting (the one-CTA kernel subtracts them
// one at a time), so results agree to rounding, not bits.
// ---------------------------------------------------------------------------
constexpr int kCholCluster = 8;
constexpr int kCholPanel = 16;
constexpr int kCholClusterMin = 64;
constexpr int kCholRows = TSVD_MAX_BLOCK / kCholCluster;  // own rows (and own columns of M) at most
constexpr int kCholLd = TSVD_MAX_BLOCK + 4, kCholLdP = kCholPanel + 1;
static_assert(kCholRows == kCholPanel && kCholPanel % kCholCluster == 0, "two own rows a panel, one lane a row");

struct CholSmem {
    double A[kCholRows][kCholLd];        // own rows of A (columns <= i), then of L
    double M[kCholRows][kCholLd];        // own rows of M (columns < i)
    double Lp[TSVD_MAX_BLOCK][kCholLdP];  // the panel's columns of L, all rows
    double Mp[kCholPanel][kCholLd];      // the panel's rows of M, all columns
    double D[kCholPanel][kCholLdP];      // the diagonal block, then its L
    double Mq[kCholPanel][kCholLdP];     // the panel's rows of M before substitution, own columns
    double col[3][32], mrow[2][kCholPanel];  // a pivot's column of L (16 + 16 rows), its row of M
    double dinv[kCholPanel];
    double thresh;
    int bad;
};

__global__ void __cluster_dims__(kCholCluster, 1, 1) __launch_bounds__(256, 1)
    chol_inv_cluster_kernel(int b, const double* __restrict__ W, double* __restrict__ Lt, double* __restrict__ Mt,
                            int* status) {
    namespace cg = cooperative_groups;
    constexpr int C = kCholCluster, P = kCholPanel;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    extern __shared__ __align__(16) unsigned char chol_raw[];
    CholSmem& sm = *reinterpret_cast<CholSmem*>(chol_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tr = tid >> 4, tx = tid & 15;       // own row and column group in the updates
    const int ti = rank + C * tr;                 // that row
    for (int idx = tid; idx < kCholRows * kCholLd; idx += 256) {
        const int r = idx / kCholLd, k = idx % kCholLd, i = rank + C * r;
        sm.A[r][k] = i < b && k <= i ? W[(size_t)i * b + k] : 0.0;
        sm.M[r][k] = 0.0;
    }
    {
        const int i = tid >> 4, k = tid & 15;  // b >= 64: the first block is whole
        sm.D[i][k] = k <= i ? W[(size_t)i * b + k] : 0.0;
        sm.Mq[i][k] = 0.0;
    }
    for (int row = rank; row < b; row += C)  // zeros left of the panel that holds the diagonal
        for (int j = tid; j < row / P * P; j += 256) {
            Lt[(size_t)row * b + j] = 0.0;
            Mt[(size_t)row * b + j] = 0.0;
        }
    if (warp == 0) {  // max of the diagonal and a non-finite flag
        double wmax = 0.0;
        int bad = 0;
        for (int i = lane; i < b; i += 32) {
            const double d = W[(size_t)i * b + i];
            if (!isfinite(d)) bad = 2;
            if (d > wmax) wmax = d;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
            bad = max(bad, __shfl_xor_sync(0xffffffffu, bad, o));
        }
        if (lane == 0) {
            if (bad == 0 && !(wmax > 0.0)) bad = 1;
            sm.bad = bad;
            sm.thresh = (double)b * kEps * wmax;
        }
    }
    cl.sync();
    int bad = sm.bad;  // the same in every CTA
    for (int p0 = 0; p0 < b && bad == 0; p0 += P) {
        const int p1 = p0 + P, pw = min(P, b - p0);
        const int r1 = p1 / C;  // own rows from here on lie below the panel
        const auto pivot_sync = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };  // from both branches
        if (warp < 4) {         // 1.
            double v[4];
            const int r = lane - 16;
            const bool below = r >= r1 && rank + C * r < b;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                v[t] = lane < 16 ? sm.D[lane][warp + 4 * t] : (below ? sm.A[max(r, 0)][p0 + warp + 4 * t] : 0.0);
            const auto pivot = [&](int j, double& x) {  // by the warp of column j
                const double d = __shfl_sync(0xffffffffu, x, j);
                double y = 1.0;
                if (j < pw) {
                    const bool finite = (__double2hiint(d) & 0x7FF00000) != 0x7FF00000;
                    if (finite && __double_as_longlong(d) > __double_as_longlong(sm.thresh)) {  // both >= 0, or d < 0
                        y = rsqrt_fp64_short(d);
                    } else if (lane == 0 && sm.bad == 0) {
                        sm.bad = finite ? 1 : 2;  // the steps run on: every warp comes to every barrier
                    }
                }
                x *= y;
                sm.col[j % 3][lane] = x;
                if (lane == 0) sm.dinv[j] = y;
            };
            if (warp == 0) pivot(0, v[0]);
#pragma unroll
            for (int j = 0; j < P; ++j) {
                pivot_sync();
                const double l = sm.col[j % 3][lane];
                const bool mine = warp == ((j + 1) & 3);
                if (j + 1 < P && mine) {
                    v[(j + 1) >> 2] = fma(-l, sm.col[j % 3][j + 1], v[(j + 1) >> 2]);
                    pivot(j + 1, v[(j + 1) >> 2]);
                }
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (warp + 4 * t > j && !(mine && t == (j + 1) >> 2))
                        v[t] = fma(-l, sm.col[j % 3][warp + 4 * t], v[t]);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int k = warp + 4 * t;
                if (lane < 16)
                    sm.D[lane][k] = k <= lane ? v[t] : 0.0;
                else if (below)
                    sm.A[r][p0 + k] = v[t];
            }
        } else {                // 2.
            double m[4];
            const int w = warp - 4, u = lane & 15, c = rank + C * u;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                m[t] = c < p0 ? sm.Mq[w + 4 * t][u] : (c - p0 == w + 4 * t ? 1.0 : 0.0);
#pragma unroll
            for (int j = 0; j < P; ++j) {
                pivot_sync();
                if (j > 0) {  // the update of pivot j - 1
                    const double x = sm.mrow[(j - 1) & 1][u];
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (w + 4 * t >= j) m[t] = fma(-sm.col[(j - 1) % 3][w + 4 * t], x, m[t]);
                }
                if (w == (j & 3)) {
                    m[j >> 2] *= sm.dinv[j];
                    if (lane < 16) sm.mrow[j & 1][u] = m[j >> 2];
                }
            }
            if (lane < 16)
#pragma unroll
                for (int t = 0; t < 4; ++t) sm.Mq[w + 4 * t][u] = m[t];
        }
        __syncthreads();
        bad = sm.bad;
        if (bad) break;
        // 3. thread (tr, tx): entry tx of own row tr of L, and row tr of own column tx of M
        if (tr >= r1 && ti < b) {
            const double x = sm.A[tr][p0 + tx];
#pragma unroll
            for (int c = 0; c < C; ++c) cl.map_shared_rank(&sm.Lp[0][0], c)[ti * kCholLdP + tx] = x;
            Lt[(size_t)(p0 + tx) * b + ti] = x;
        }
        {
            const int c = rank + C * tx;
            if (c < p1 && c < b) {
                const double x = sm.Mq[tr][tx];
#pragma unroll
                for (int u = 0; u < C; ++u) cl.map_shared_rank(&sm.Mp[0][0], u)[tr * kCholLd + c] = x;
                if (p0 + tr < b) Mt[(size_t)c * b + p0 + tr] = x;
            }
        }
        if (rank == 0 && tr < pw && tx < pw) Lt[(size_t)(p0 + tx) * b + p0 + tr] = sm.D[tr][tx];
        if (p1 >= b) break;
        cl.sync();
        // 4.
        if (tr >= r1 && ti < b) {
            double li[P];
#pragma unroll
            for (int l = 0; l < P; ++l) li[l] = sm.A[tr][p0 + l];
            for (int k = tx; k < p1; k += 16) {
                double acc = 0.0;
#pragma unroll
                for (int l = 0; l < P; ++l) acc = fma(li[l], sm.Mp[l][k], acc);
                sm.M[tr][k] -= acc;
            }
            for (int k = p1 + tx; k <= ti; k += 16) {
                double acc = 0.0;
#pragma unroll
                for (int l = 0; l < P; ++l) acc = fma(li[l], sm.Lp[k][l], acc);
                sm.A[tr][k] -= acc;
            }
        }
        __syncthreads();
        {  // the two own rows of the next panel
            const int half = tid >> 7, e = tid & 127, r = r1 + half, i = rank + C * r;
            const bool in = r < kCholRows && i < b;
            // diagonal block: entry e / 8 for CTA e % 8
            const int k = e >> 3;
            if (r < kCholRows)
                cl.map_shared_rank(&sm.D[0][0], e & 7)[(i - p1) * kCholLdP + k] = in && p1 + k <= i ? sm.A[r][p1 + k] : 0.0;
            // M: column e to its owner
            if (r < kCholRows && e < p1)
                cl.map_shared_rank(&sm.Mq[0][0], e & 7)[(i - p1) * kCholLdP + (e >> 3)] = in ? sm.M[r][e] : 0.0;
        }
        cl.sync();
    }
    // (the copies of one's rows end at a barrier; after a last panel nobody writes to another CTA's
    // memory but in step 3, so wait for that too)
    cl.sync();
    if (bad) {
        if (rank == 0 && tid == 0) atomicOr(&status[bad == 2 ? kStNonfinite : kStBreakdown], 1);
        for (int idx = rank * 256 + tid; idx < b * b; idx += C * 256) {
            const double v = (idx / b == idx % b) ? 1.0 : 0.0;
            Lt[idx] = v;
            Mt[idx] = v;
        }
    }
}

// out = A U, A and U upper triangular b x b (ld b).  Block = one row i.
__global__ void trmm_upper_kernel(int b, const double* __restrict__ A, const double* __restrict__ U,
                                  double* __restrict__ out, int64_t ldo, int trans) {
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < b; j += blockDim.x) {
        double acc = 0.0;
        for (int k = i; k <= j; ++k) acc = fma(A[i * b + k], U[k * b + j], acc);
        if (trans)
            out[(int64_t)j * ldo + i] = acc;
        else
            out[(int64_t)i * ldo + j] = acc;
    }
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11) and Box-Muller.
// ---------------------------------------------------------------------------
__device__ inline void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
        const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
    }
}

__global__ void gaussian_kernel(int64_t rows, int64_t cols, uint32_t k0, uint32_t k1, uint32_t sid,
                                double* __restrict__ out, int64_t ld, int64_t e_off) {
    // elements e_off .. e_off + rows cols - 1 of the row-major global block: element e
    // is half of Philox counter e / 2, so a slice that starts at an odd element drops
    // the first half of its first pair
    const int64_t n_el = rows * cols;
    const int64_t t0 = e_off / 2, t1 = (e_off + n_el - 1) / 2;
    for (int64_t t = t0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= t1;
         t += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c[4] = {(uint32_t)(t & 0xffffffffu), (uint32_t)((uint64_t)t >> 32), sid, 0u};
        philox4x32_10(c, k0, k1);
        const double two53 = 1.1102230246251565e-16;  // 2^-53
        const double u1 = (double)(((uint64_t)(c[0] >> 5) << 26) + (c[1] >> 6) + 1) * two53;
        const double u2 = (double)(((uint64_t)(c[2] >> 5) << 26) + (c[3] >> 6) + 1) * two53;
        const double rad = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        const int64_t e0 = 2 * t - e_off, e1 = e0 + 1;
        if (e0 >= 0 && e0 < n_el) out[(e0 / cols) * ld + (e0 % cols)] = rad * cs;
        if (e1 >= 0 && e1 < n_el) out[(e1 / cols) * ld + (e1 % cols)] = rad * sn;
    }
}

// ---------------------------------------------------------------------------
// Residual column sums of squares, Lanczos estimate, sign convention.
// ---------------------------------------------------------------------------
// (Blocks of 32 columns x 8 rows: the rows of a group are split over the block, as in
// coldot.  With one thread a column, residual norms of 100,000 x 64 took 170 us and the
// largest entries of its columns 165 us, against 30 us and 25 us.)
__global__ void __launch_bounds__(256)
    colres_partial_kernel(int64_t q, int k, const double* __restrict__ Y, int64_t ldy, const double* __restrict__ U,
                          int64_t ldu, const double* __restrict__ sigma, double* __restrict__ partial,
                          int64_t rows_per) {
    __shared__ double red[8][33];
    const int64_t r0 = (int64_t)blockIdx.x * rows_per, r1 = min(q, r0 + rows_per);
    const int j = (int)blockIdx.y * 32 + threadIdx.x;
    double acc = 0.0;
    if (j < k) {
        const double sj = sigma[j];
#pragma unroll 4
        for (int64_t i = r0 + threadIdx.y; i < r1; i += 8) {
            const double d = fma(-U[i * ldu + j], sj, Y[i * ldy + j]);
            acc = fma(d, d, acc);
        }
    }
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && j < k) {
#pragma unroll
        for (int y = 1; y < 8; ++y) acc += red[y][threadIdx.x];
        partial[(int64_t)blockIdx.x * k + j] = acc;
    }
}

// out[j] = sum_g partial[g][j]: thread (x, y) adds groups y, y + 32, .. of column x, then
// the 32 sums are added in order.
__global__ void __launch_bounds__(1024) col_sum_kernel(int k, int g, const double* __restrict__ partial,
                                                       double* __restrict__ out) {
    __shared__ double red[32][33];
    const int j = (int)blockIdx.x * 32 + threadIdx.x;
    double acc = 0.0;
    if (j < k)
        for (int t = threadIdx.y; t < g; t += 32) acc += partial[(int64_t)t * k + j];
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && j < k) {
        for (int y = 1; y < 32; ++y) acc += red[y][threadIdx.x];
        out[j] = acc;
    }
}

// rho[j], one block a column: y = Rr v_j with a warp a row, then the sum of squares in row
// order.  (One block for all columns took 0.70 ms at b = 128, k = 100; 8 us now.)
__global__ void __launch_bounds__(256) lanczos_rho_kernel(int b, int k, const double* __restrict__ Rr,
                                                          const double* __restrict__ V, int64_t ldv,
                                                          double* __restrict__ rho) {
    __shared__ double v[TSVD_MAX_BLOCK], y2[TSVD_MAX_BLOCK];
    const int j = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l = threadIdx.x; l < b; l += blockDim.x) v[l] = V[(int64_t)l * ldv + j];
    __syncthreads();
    for (int i = warp; i < b; i += (int)blockDim.x >> 5) {
        double yi = 0.0;
        for (int l = i + lane; l < b; l += 32) yi = fma(Rr[i * b + l], v[l], yi);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) yi += __shfl_xor_sync(0xffffffffu, yi, o);
        if (lane == 0) y2[i] = yi * yi;
    }
    __syncthreads();
    if (warp == 0) {
        double acc = 0.0;
        for (int i = lane; i < b; i += 32) acc += y2[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) rho[j] = sqrt(acc);
    }
}

// The larger magnitude wins, the smaller row on ties.
__device__ inline void argmax_take(double& best, int64_t& bi, double a, int64_t i) {
    if (a > best || (a == best && i < bi)) {
        best = a;
        bi = i;
    }
}

__global__ void __launch_bounds__(256)
    argmax_partial_kernel(int64_t n, int k, const double* __restrict__ V, int64_t ldv, int64_t rows_per,
                          double* __restrict__ pv, int64_t* __restrict__ pi) {
    __shared__ double sv[8][33];
    __shared__ int64_t si[8][33];
    const int64_t r0 = (int64_t)blockIdx.x * rows_per, r1 = min(n, r0 + rows_per);
    const int j = (int)blockIdx.y * 32 + threadIdx.x;
    double best = -1.0;
    int64_t bi = 0;
    if (j < k) {
#pragma unroll 4
        for (int64_t i = r0 + threadIdx.y; i < r1; i += 8) {
            const double a = fabs(V[i * ldv + j]);
            if (a > best) {
                best = a;
                bi = i;
            }
        }
    }
    sv[threadIdx.y][threadIdx.x] = best;
    si[threadIdx.y][threadIdx.x] = bi;
    __syncthreads();
    if (threadIdx.y == 0 && j < k) {
#pragma unroll
        for (int y = 1; y < 8; ++y) argmax_take(best, bi, sv[y][threadIdx.x], si[y][threadIdx.x]);
        pv[(int64_t)blockIdx.x * k + j] = best;
        pi[(int64_t)blockIdx.x * k + j] = bi;
    }
}

__global__ void __launch_bounds__(1024)
    argmax_sign_kernel(int k, int g, const double* __restrict__ pv, const int64_t* __restrict__ pi,
                       const double* __restrict__ V, int64_t ldv, double* __restrict__ sgn) {
    __shared__ double sv[32][33];
    __shared__ int64_t si[32][33];
    const int j = (int)blockIdx.x * 32 + threadIdx.x;
    double best = -1.0;
    int64_t bi = 0;
    if (j < k)
        for (int t = threadIdx.y; t < g; t += 32)
            argmax_take(best, bi, pv[(int64_t)t * k + j], pi[(int64_t)t * k + j]);
    sv[threadIdx.y][threadIdx.x] = best;
    si[threadIdx.y][threadIdx.x] = bi;
    __syncthreads();
    if (threadIdx.y == 0 && j < k) {
        for (int y = 1; y < 32; ++y) argmax_take(best, bi, sv[y][threadIdx.x], si[y][threadIdx.x]);
        sgn[j] = V[bi * ldv + j] < 0.0 ? -1.0 : 1.0;
    }
}

__global__ void apply_sign_kernel(int64_t rows, int k, double* __restrict__ A, int64_t lda,
                                  const double* __restrict__ sgn) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * k) return;
    const int64_t i = idx / k;
    const int j = (int)(idx % k);
    if (sgn[j] < 0.0) A[i * lda + j] = -A[i * lda + j];
}

__global__ void put_transposed_kernel(int rows, int cols, const double* __restrict__ H, int64_t ldh,
                                      double* __restrict__ D, int64_t ldd) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)rows * cols) return;
    const int i = (int)(idx / cols), j = (int)(idx % cols);
    D[(int64_t)j * ldd + i] = H[(int64_t)i * ldh + j];
}

__global__ void put_diagonal_kernel(int s, const double* __restrict__ sig, double* __restrict__ B, int64_t ldb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < s) B[(int64_t)i * ldb + i] = sig[i];
}

}  // namespace

// ---------------------------------------------------------------------------
size_t gemm_tn_ws(tsvd_handle* h, int64_t q, int64_t s, int64_t b, bool symmetric, int elem_bytes) {
    const size_t least = gemm_tn_ws_min(h, q, s, b, symmetric, elem_bytes);
    return elem_bytes == 8 ? std::max(least, kTnExtra) : least;
}
size_t gemm_tn_ws_min(tsvd_handle* h, int64_t q, int64_t s, int64_t b, bool symmetric, int elem_bytes) {
    (void)h;
    const TnPlan p = tn_plan(q, s, b, symmetric, elem_bytes, false);
    if (p.slabs == 1 && !symmetric) return 0;
    return align256(sizeof(double) * (size_t)p.slabs * (size_t)s * (size_t)b);
}

size_t gemm_tn_ws_bound(int64_t q, int64_t s, int64_t b, bool symmetric, int elem_bytes) {
    const int64_t wave = elem_bytes == 4 ? kTnWaveF32 : kTnWave;
    const int64_t max_slabs = std::max<int64_t>(1, std::min<int64_t>((q + 255) / 256, 65535));
    int64_t most = 0;  // doubles
    for (int64_t i = 1; i <= (s + kTnR - 1) / kTnR; ++i)
        for (int64_t j = symmetric ? i : 1; j <= (symmetric ? i : (b + kTnR - 1) / kTnR); ++j) {
            const int64_t regions = symmetric ? i * (i + 1) / 2 : i * j;
            const int64_t slabs = std::max<int64_t>(1, std::min(wave / regions, max_slabs));
            most = std::max(most, slabs * std::min(s, i * kTnR) * std::min(b, j * kTnR));
        }
    return std::max(align256(sizeof(double) * (size_t)most), elem_bytes == 8 ? kTnExtra : 0);
}

template <typename TI, typename TC>
cudaError_t gemm_tn(tsvd_handle* h, int64_t q, int64_t s, int64_t b, const TI* X, int64_t ldx, const TI* Z,
                    int64_t ldz, TC* C, int64_t ldc, bool symmetric, double* partial, cudaStream_t st,
                    size_t partial_bytes, bool fp64_pipe) {
    if (s == 0 || b == 0) return cudaSuccess;
    constexpr bool kF32 = std::is_same<TI, float>::value;
    const TnPlan p = tn_plan(q, s, b, symmetric, (int)sizeof(TI), partial_bytes >= kTnExtra);
    if (q == 0) {
        for (int64_t i = 0; i < s; ++i) {
            cudaError_t e = cudaMemsetAsync(C + i * ldc, 0, sizeof(TC) * b, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    dim3 grid((unsigned)p.regions, (unsigned)p.slabs);
    // algorithmic work: 2qsb flops (the upper half, q b (b+1), for a Gram matrix);
    // compulsory traffic: X and Z read once, C written once
    ProfScope prof(h, TSVD_K_GEMM_TN, symmetric ? (double)q * b * (b + 1) : 2.0 * q * s * b,
                   (double)sizeof(TI) * (double)q * (symmetric ? b : s + b) + (double)sizeof(TC) * s * b, st);
    if constexpr (std::is_same<TI, double>::value && std::is_same<TC, double>::value) {
        const OzCache* xc = h->oz_ws ? oz_find_cache(h, X, ldx, q, s, true) : nullptr;
        if (!fp64_pipe && h->oz_ws && oz_worth(s, b, q) && oz_tn_ws(q, s, b, symmetric, xc != nullptr, h->oz_dig) <= h->oz_bytes) {
            const int rc = oz_gemm_tn(h, q, s, b, X, ldx, Z, ldz, C, ldc, symmetric, h->oz_ws, h->oz_bytes,
                                      h->oz_status, st, xc);
            return rc == TSVD_OK ? cudaSuccess : cudaErrorUnknown;
        }
    }
    int slabs = p.slabs;
    int64_t slab_rows = p.slab_rows;
    bool wide = false;
    if constexpr (kF32) {
        // one CTA an SM, in no more slabs than the partial sums have room for
        const int regions = symmetric ? 0 : wide_f32_regions(q, s, b);
        wide = regions > 0;
        if (wide) {
            // (two waves where a thread would otherwise add up more rows in FP32 than in the
            // other kernel's plan: for b <= 64 and regions that are not full; 500,003 x 96 by 64:
            // 233 us and 5.2e-7 off, in one wave 220 us and 7.3e-7, the other kernel 377 us and 6.3e-7)
            const int wave = std::max(1, 152 / regions);
            const bool long_runs = 2 * (int64_t)wave < p.slabs;
            slabs = std::min(slabs, long_runs ? 2 * wave : wave);
            slab_rows = ((q + slabs - 1) / slabs + 31) / 32 * 32;
            slabs = (int)((q + slab_rows - 1) / slab_rows);
            grid = dim3((unsigned)regions, (unsigned)slabs);
        }
    }
    if (slabs == 1 && !symmetric) {
        h->launches++;
        if constexpr (kF32)
            if (wide) return launch_gemm_tn_wide_f32<TC>(grid, st, q, s, b, X, ldx, Z, ldz, C, ldc, 0, slab_rows);
        if constexpr (kF32)
            return launch_gemm_tn_f32<TC>(grid, st, q, s, b, X, ldx, Z, ldz, C, ldc, 0, p.slab_rows, 0, p.nreg_s,
                                          p.nreg_b);
        gemm_tn_kernel<TI, TC><<<grid, 128, 0, st>>>(q, s, b, X, ldx, Z, ldz, C, ldc, 0, p.slab_rows, 0, p.nreg_s,
                                                     p.nreg_b);
        return cudaGetLastError();
    }
    const int64_t stride = s * b;
    h->launches += 2;
    if constexpr (kF32) {
        cudaError_t e = wide ? launch_gemm_tn_wide_f32<double>(grid, st, q, s, b, X, ldx, Z, ldz, partial, b, stride,
                                                               slab_rows)
                             : launch_gemm_tn_f32<double>(grid, st, q, s, b, X, ldx, Z, ldz, partial, b, stride, p.slab_rows,
                                                   symmetric ? 1 : 0, p.nreg_s, p.nreg_b);
        if (e != cudaSuccess) return e;
    } else {
        gemm_tn_kernel<TI, double><<<grid, 128, 0, st>>>(q, s, b, X, ldx, Z, ldz, partial, b, stride, p.slab_rows,
                                                         symmetric ? 1 : 0, p.nreg_s, p.nreg_b);
    }
    const int64_t tot = s * b;
    gemm_tn_reduce_kernel<TC><<<(unsigned)((tot + 31) / 32), dim3(32, 8), 0, st>>>(s, b, slabs, partial, stride, C,
                                                                                  ldc, symmetric ? 1 : 0);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Fused update + Gram of FP32 blocks.  One CTA per slab of consecutive 64-row
// tiles; the split targets one wave of the kernel's resident 256-thread CTAs on
// 152 SMs: 4 per SM for b <= 64, 2 for b <= 128 (a fixed target, so the split, the
// workspace and the summation order do not depend on the device).
struct UgPlan {
    int slabs;
    int64_t slab_rows;
};

static UgPlan ug_plan(int64_t q, int64_t b) {
    UgPlan p;
    const int64_t wave = 152 * (b <= 64 ? 4 : 2);
    int64_t tiles = (q + 63) / 64;
    if (tiles < 1) tiles = 1;
    const int64_t slabs = tiles < wave ? tiles : wave;
    p.slab_rows = (tiles + slabs - 1) / slabs * 64;
    p.slabs = (int)((q + p.slab_rows - 1) / p.slab_rows);
    if (p.slabs < 1) p.slabs = 1;
    return p;
}

size_t update_gram_ws(int64_t q, int64_t b) {
    return align256(sizeof(double) * (size_t)ug_plan(q, b).slabs * (size_t)b * (size_t)b);
}

cudaError_t update_gram(tsvd_handle* h, int64_t q, int64_t s, int64_t b, double alpha, const float* X, int64_t ldx,
                        const double* M, int64_t ldm, double beta, float* Y, int64_t ldy, bool upper, double* W,
                        double* partial, cudaStream_t st) {
    if (b < 1 || b > 128 || s < 1) return cudaErrorInvalidValue;
    if (q == 0) return cudaMemsetAsync(W, 0, sizeof(double) * (size_t)b * b, st);
    const UgPlan p = ug_plan(q, b);
    // algorithmic work: the update (2qsb, or q b (b+1) for a triangular M) plus the
    // upper half of the Gram matrix, q b (b+1); compulsory traffic: X and M read,
    // Y read (beta != 0, unless it is X) and written, W written
    const bool alias = (const void*)X == (const void*)Y;
    const double upd = upper ? (double)q * b * (b + 1) : 2.0 * q * s * b;
    const double bytes = 4.0 * q * s + ((beta != 0.0 && !alias) ? 4.0 * q * b : 0.0) + 4.0 * q * b +
                         8.0 * s * b + 8.0 * b * b;
    ProfScope prof(h, TSVD_K_UPD_GRAM, upd + (double)q * b * (b + 1), bytes, st);
    h->launches += 2;
    cudaError_t e = launch_update_gram_f32<double>(st, p.slabs, p.slab_rows, q, s, b, alpha, X, ldx, M, ldm, beta, Y,
                                                   ldy, upper, partial);
    if (e != cudaSuccess) return e;
    gemm_tn_reduce_kernel<double><<<(unsigned)((b * b + 31) / 32), dim3(32, 8), 0, st>>>(b, b, p.slabs, partial,
                                                                                         b * b, W, b, 1);
    return cudaGetLastError();
}

template cudaError_t gemm_tn<double, double>(tsvd_handle*, int64_t, int64_t, int64_t, const double*, int64_t,
                                             const double*, int64_t, double*, int64_t, bool, double*, cudaStream_t, size_t, bool);
template cudaError_t gemm_tn<float, double>(tsvd_handle*, int64_t, int64_t, int64_t, const float*, int64_t,
                                            const float*, int64_t, double*, int64_t, bool, double*, cudaStream_t, size_t, bool);
template cudaError_t gemm_tn<float, float>(tsvd_handle*, int64_t, int64_t, int64_t, const float*, int64_t,
                                           const float*, int64_t, float*, int64_t, bool, double*, cudaStream_t, size_t, bool);

template <typename TX, typename TM, typename TY>
cudaError_t gemm_nn(tsvd_handle* h, int64_t q, int64_t s, int64_t b, double alpha, const TX* X, int64_t ldx,
                    const TM* M, int64_t ldm, double beta, TY* Y, int64_t ldy, bool upper, cudaStream_t st,
                    bool fp64_pipe) {
    if (q == 0 || b == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((q + 31) / 32);
    ProfScope prof(h, TSVD_K_GEMM_NN, upper ? (double)q * b * (b + 1) : 2.0 * q * s * b,
                   (double)sizeof(TX) * q * s + (double)sizeof(TM) * s * b +
                       (double)sizeof(TY) * q * b * (beta != 0.0 ? 2 : 1), st);
    if constexpr (std::is_same<TX, double>::value && std::is_same<TM, double>::value &&
                  std::is_same<TY, double>::value) {
        const OzCache* xc = h->oz_ws && !h->oz_fresh_rows ? oz_find_cache(h, X, ldx, q, s, false) : nullptr;
        if (!fp64_pipe && h->oz_ws && s > 0 && oz_worth(q, b, s) && oz_nn_ws(q, s, b, xc != nullptr, h->oz_dig) <= h->oz_bytes) {
            const int rc = oz_gemm_nn(h, q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, upper, h->oz_ws, h->oz_bytes,
                                      h->oz_status, st, xc);
            return rc == TSVD_OK ? cudaSuccess : cudaErrorUnknown;
        }
    }
    h->launches++;
    if constexpr (std::is_same<TX, float>::value) {
        if (b <= 128) return launch_gemm_nn_f32<TM, TY>(st, q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, upper);
    }
    // Columns of a CTA: all of them (up to 128) where X is read from memory once that way;
    // fewer while the grid leaves SMs without a CTA (the FP64 pipe of an SM then bounds the
    // time: 512 x 64 by 64 x 16 took 31 us on 16 SMs), but not in place, where one CTA reads
    // all of its rows before it writes them.
    int cw = b <= 16 ? 4 : (b <= 32 ? 8 : (b <= 64 ? 16 : 32));
    if constexpr (!std::is_same<TX, double>::value) cw = std::max(cw, 8);
    const uintptr_t x0 = reinterpret_cast<uintptr_t>(X), x1 = reinterpret_cast<uintptr_t>(X + q * ldx);
    const uintptr_t y0 = reinterpret_cast<uintptr_t>(Y), y1 = reinterpret_cast<uintptr_t>(Y + q * ldy);
    unsigned gy = 1;
    if (std::is_same<TX, double>::value && (x1 <= y0 || y1 <= x0)) {
        while (cw > 1 && (int64_t)grid * ((b + 4 * cw - 1) / (4 * cw)) < 152) cw /= 2;
        if ((int64_t)grid < 152) gy = (unsigned)std::min<int64_t>((b + 4 * cw - 1) / (4 * cw), 65535);
    }
    const dim3 g(grid, gy);
    const int up = upper ? 1 : 0;
    if (cw == 32) {
        gemm_nn_kernel<32, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
    } else if (cw == 16) {
        gemm_nn_kernel<16, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
    } else if (cw == 8) {
        gemm_nn_kernel<8, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
    } else if constexpr (std::is_same<TX, double>::value) {
        if (cw == 4)
            gemm_nn_kernel<4, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
        else if (cw == 2)
            gemm_nn_kernel<2, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
        else
            gemm_nn_kernel<1, TX, TM, TY><<<g, 128, 0, st>>>(q, s, b, alpha, X, ldx, M, ldm, beta, Y, ldy, up);
    }
    return cudaGetLastError();
}

#define TSVD_INST_NN(TX, TM, TY)                                                                                  \
    template cudaError_t gemm_nn<TX, TM, TY>(tsvd_handle*, int64_t, int64_t, int64_t, double, const TX*, int64_t, \
                                             const TM*, int64_t, double, TY*, int64_t, bool, cudaStream_t, bool);
TSVD_INST_NN(double, double, double)
TSVD_INST_NN(float, double, float)
TSVD_INST_NN(float, float, float)
TSVD_INST_NN(float, double, double)
#undef TSVD_INST_NN

static size_t chol_smem(int b) { return sizeof(double) * ((size_t)b * (b + 1) + b); }

cudaError_t chol_inv(tsvd_handle* h, int b, const double* W, double* Lt, double* Mt, int* status,
                     cudaStream_t st) {
    const size_t smem = chol_smem(b);
    static thread_local int configured_device = -1;
    if (configured_device != h->device) {
        cudaError_t e = cudaFuncSetAttribute(chol_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)chol_smem(kCholClusterMin - 1));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(chol_inv_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(CholSmem));
        if (e != cudaSuccess) return e;
        configured_device = h->device;
    }
    ProfScope prof(h, TSVD_K_CHOL, 2.0 * b * b * (double)b / 3.0, 24.0 * b * b, st);
    h->launches++;
    if (b >= kCholClusterMin)
        chol_inv_cluster_kernel<<<kCholCluster, 256, sizeof(CholSmem), st>>>(b, W, Lt, Mt, status);
    else
        chol_inv_kernel<<<1, 256, smem, st>>>(b, W, Lt, Mt, status);
    return cudaGetLastError();
}

cudaError_t trmm_upper(tsvd_handle* h, int b, const double* A, const double* U, double* out, int64_t ldo,
                       bool trans, cudaStream_t st) {
    ProfScope prof(h, TSVD_K_OTHER, b * b * (double)b / 3.0, 24.0 * b * b, st);
    h->launches++;
    trmm_upper_kernel<<<b, 128, 0, st>>>(b, A, U, out, ldo, trans ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t gaussian(tsvd_handle* h, int64_t rows, int64_t cols, uint64_t seed, uint32_t stream_id, double* out,
                     int64_t ld, cudaStream_t st, int64_t row0) {
    if (rows * cols == 0) return cudaSuccess;
    const int64_t e_off = row0 * cols;
    const int64_t n_pairs = (e_off + rows * cols - 1) / 2 - e_off / 2 + 1;
    int64_t blocks = (n_pairs + 255) / 256;
    if (blocks > 8LL * h->sm_count * 8) blocks = 8LL * h->sm_count * 8;
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 8.0 * rows * cols, st);
    h->launches++;
    gaussian_kernel<<<(unsigned)blocks, 256, 0, st>>>(rows, cols, (uint32_t)(seed & 0xffffffffu),
                                                      (uint32_t)(seed >> 32), stream_id, out, ld, e_off);
    return cudaGetLastError();
}

size_t colres_ws(int64_t q, int k) { return align256(sizeof(double) * (size_t)col_groups(q) * (size_t)k); }

cudaError_t col_sum(tsvd_handle* h, int groups, int k, const double* partial, double* out, cudaStream_t st) {
    h->launches++;
    col_sum_kernel<<<(unsigned)((k + 31) / 32), dim3(32, 32), 0, st>>>(k, groups, partial, out);
    return cudaGetLastError();
}

cudaError_t col_residual_sq(tsvd_handle* h, int64_t q, int k, const double* Y, int64_t ldy, const double* U,
                            int64_t ldu, const double* sigma, double* out, double* partial, cudaStream_t st) {
    const int g = col_groups(q);
    const int64_t rows_per = (q + g - 1) / g;
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 0.0, st);
    h->launches++;
    colres_partial_kernel<<<dim3((unsigned)g, (unsigned)((k + 31) / 32)), dim3(32, 8), 0, st>>>(
        q, k, Y, ldy, U, ldu, sigma, partial, rows_per);
    return col_sum(h, g, k, partial, out, st);
}

cudaError_t put_transposed(tsvd_handle* h, int rows, int cols, const double* H, int64_t ldh, double* D, int64_t ldd,
                           cudaStream_t st) {
    if (rows == 0 || cols == 0) return cudaSuccess;
    const int64_t tot = (int64_t)rows * cols;
    h->launches++;
    put_transposed_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(rows, cols, H, ldh, D, ldd);
    return cudaGetLastError();
}

cudaError_t put_diagonal(tsvd_handle* h, int s, const double* sig, double* B, int64_t ldb, cudaStream_t st) {
    if (s == 0) return cudaSuccess;
    h->launches++;
    put_diagonal_kernel<<<(unsigned)((s + 255) / 256), 256, 0, st>>>(s, sig, B, ldb);
    return cudaGetLastError();
}

cudaError_t lanczos_rho(tsvd_handle* h, int b, int k, const double* Rr, const double* Vlast, int64_t ldv,
                        double* rho, cudaStream_t st) {
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 0.0, st);
    h->launches++;
    lanczos_rho_kernel<<<k, 256, 0, st>>>(b, k, Rr, Vlast, ldv, rho);
    return cudaGetLastError();
}

size_t sign_fix_ws(int64_t n, int k) {
    const size_t g = (size_t)col_groups(n);
    return align256(sizeof(double) * g * k) + align256(sizeof(int64_t) * g * k) + align256(sizeof(double) * k);
}

cudaError_t sign_fix(tsvd_handle* h, int64_t n, int64_t m, int k, double* V, int64_t ldv, double* U, int64_t ldu,
                     void* ws, cudaStream_t st) {
    const int g = col_groups(n);
    char* p = static_cast<char*>(ws);
    double* pv = reinterpret_cast<double*>(p);
    p += align256(sizeof(double) * (size_t)g * k);
    int64_t* pi = reinterpret_cast<int64_t*>(p);
    p += align256(sizeof(int64_t) * (size_t)g * k);
    double* sgn = reinterpret_cast<double*>(p);
    const int64_t rows_per = (n + g - 1) / g;
    ProfScope prof(h, TSVD_K_OTHER, 0.0, 0.0, st);
    h->launches += 4;
    const unsigned strips = (unsigned)((k + 31) / 32);
    argmax_partial_kernel<<<dim3((unsigned)g, strips), dim3(32, 8), 0, st>>>(n, k, V, ldv, rows_per, pv, pi);
    argmax_sign_kernel<<<strips, dim3(32, 32), 0, st>>>(k, g, pv, pi, V, ldv, sgn);
    if (n * k > 0) apply_sign_kernel<<<(unsigned)((n * k + 255) / 256), 256, 0, st>>>(n, k, V, ldv, sgn);
    if (m * k > 0) apply_sign_kernel<<<(unsigned)((m * k + 255) / 256), 256, 0, st>>>(m, k, U, ldu, sgn);
    return cudaGetLastError();
}

}  // namespace tsvd
