// Small SVD of the projected matrix (R_p of Alg. 1 S5, B_k of Alg. 2 S6) on the
// device: one-sided Jacobi (Hestenes 1958) on the columns of B, with the
// parallel round-robin ("tournament") pair ordering of Brent and Luk (1985) so
// that n/2 disjoint column pairs rotate at once.  The paper runs this step as
// LAPACK GESVD on the host; here it stays on the GPU so the iteration never
// leaves the device.
//
// Layout: G = B padded to an even number of columns with a zero column,
// column-major (ld = n rows); V = identity of order npad, column-major.  One
// warp owns one pair per round: it forms alpha = |g_p|^2, beta = |g_q|^2,
// gamma = g_p.g_q with a fixed shuffle tree, and if |gamma| > tol*sqrt(alpha*beta)
// applies the rotation with t = sign(zeta)/(|zeta| + hypot(1, zeta)),
// zeta = (beta - alpha)/(2 gamma) (Rutishauser's formulas) to both G and V.
// Rounds are separated by a grid barrier whose wait is bounded (clock64, ~1 s):
// on timeout it raises the status word and every CTA returns.  Sweeps repeat until one sweep
// rotates nothing (or kMaxSweeps).  Then sigma_j = |g_j|, columns are sorted by
// (sigma descending, index ascending), Ubar_j = g_j / sigma_j, Vbar_j = v_j, and
// each pair is sign-flipped so the largest-magnitude entry of Vbar_j is positive.
#include <cooperative_groups.h>

#include <algorithm>

#include "tsvd_internal.cuh"

namespace tsvd {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxSweeps = 40;

enum Ctl : int { kCtlCount = 0, kCtlErr = 1, kCtlSweeps = 3, kCtlVBad = 4, kCtlNeed = 5, kCtlRot = 8 };
constexpr int kCtlWords = kCtlRot + kMaxSweeps;

__device__ inline unsigned vload(const unsigned* p) { return *reinterpret_cast<const volatile unsigned*>(p); }

__device__ inline void arrive_release(unsigned* p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ inline unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Words 0 and 1 at p (8-byte aligned), read together.
__device__ inline uint2 load2_acquire(const unsigned* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return make_uint2((unsigned)v, (unsigned)(v >> 32));
}

// Grid-wide barrier for a cooperative launch (all CTAs co-resident): a count that only grows,
// `epoch` times gridDim.x once every CTA has come (kept by each CTA, 0 at the start); one wait
// gives up after max_wait SM clock cycles (the handle's limit, about 1 s by default).
// Returns false once any CTA has timed out; the answer is read once per CTA (by thread 0,
// through shared memory), so every thread of a CTA takes the same branch and none is left at
// a later __syncthreads.  (A count that the last CTA resets, with a generation word to release
// the others, added two more trips to memory to every barrier.)
__device__ bool grid_sync(unsigned* ctl, long long max_wait, unsigned& epoch) {
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    __shared__ int s_ok;
    __syncthreads();
    ++epoch;
    if (threadIdx.x == 0) {
        arrive_release(&ctl[kCtlCount]);
        // busy-wait (naps wake late), bounded by the SM clock
        const long long t0 = clock64();
        uint2 v;  // count and error word in one read
        while (v = load2_acquire(ctl), v.x < epoch * gridDim.x) {
            if (clock64() - t0 > max_wait) {
                atomicOr(&ctl[kCtlErr], 1u);
                v.y = 1u;
                break;
            }
        }
        s_ok = v.y == 0u ? 1 : 0;
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ inline double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
    return v;
}

// Player at seat `seat` in round `rnd` of the round-robin on npad players.
__device__ inline int rr_player(int seat, int rnd, int npad) {
    return seat == 0 ? 0 : ((seat - 1 + rnd) % (npad - 1)) + 1;
}

__global__ void jacobi_init_kernel(int n, int npad, const double* __restrict__ B, int64_t ldb,
                                   double* __restrict__ G, double* __restrict__ V) {
    const int64_t tot = (int64_t)npad * npad;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(idx / npad), r = (int)(idx % npad);
        V[idx] = (c == r) ? 1.0 : 0.0;
        if (r < n) G[(int64_t)c * n + r] = (c < n) ? B[(int64_t)r * ldb + c] : 0.0;
    }
}

constexpr int kJWarps = 4;     // warps per CTA when several CTAs share the sweep
constexpr int kMaxSlots = 64;  // column pairs one CTA owns per round

// One-sided Jacobi sweeps.  CTA b owns the round's pairs [b*ppb, (b+1)*ppb).
// Per round: (A) each warp forms gamma = g_p.g_q for its pairs; (B) one lane per
// pair turns (alpha, beta, gamma) into the rotation (c, s) and updates the squared
// column norms alpha - t*gamma, beta + t*gamma (exact consequences of the rotation;
// recomputed exactly at every sweep start); (C) the warps apply the rotations to
// G (and to V when it is accumulated).  A warp-wide FP64 instruction costs the
// 2-lane FP64 pipe the same whatever its active lanes, so the scalar work of (B)
// is done once per pair, and its divide and square roots run in FP32 (see (B)).
__global__ void jacobi_sweep_kernel(int n, int npad, double* __restrict__ G, double* __restrict__ V,
                                    double* __restrict__ nrm, unsigned* ctl, double tol, int ppb,
                                    long long max_wait) {
    const double tol2 = tol * tol;
    unsigned epoch = 0;
    __shared__ double s_gam[kMaxSlots], s_c[kMaxSlots], s_s[kMaxSlots];
    __shared__ int s_rot[kMaxSlots];
    __shared__ int s_any;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    const int npairs = npad / 2;
    const int base = blockIdx.x * ppb;
    const int cnt = max(0, min(ppb, npairs - base));
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        // exact squared column norms at the start of the sweep
        for (int c = blockIdx.x * wpb + warp; c < npad; c += gridDim.x * wpb) {
            const double* g = G + (int64_t)c * n;
            double acc = 0.0;
            for (int r = lane; r < n; r += 32) acc = fma(g[r], g[r], acc);
            acc = warp_sum(acc);
            if (lane == 0) nrm[c] = acc;
        }
        if (threadIdx.x == 0) s_any = 0;
        if (!grid_sync(ctl, max_wait, epoch)) return;
        for (int rnd = 0; rnd < npad - 1; ++rnd) {
            for (int slot = warp; slot < cnt; slot += wpb) {                     // (A)
                const int pi = base + slot;
                const int a = rr_player(pi, rnd, npad), bq = rr_player(npad - 1 - pi, rnd, npad);
                const double* gp = G + (int64_t)min(a, bq) * n;
                const double* gq = G + (int64_t)max(a, bq) * n;
                double ga = 0.0;
                for (int r = lane; r < n; r += 32) ga = fma(gp[r], gq[r], ga);
                ga = warp_sum(ga);
                if (lane == 0) s_gam[slot] = ga;
            }
            __syncthreads();
            if (warp == 0) {                                                      // (B)
                for (int slot = lane; slot < cnt; slot += 32) {
                    const int pi = base + slot;
                    const int a = rr_player(pi, rnd, npad), bq = rr_player(npad - 1 - pi, rnd, npad);
                    const int p = min(a, bq), q = max(a, bq);
                    const double al = nrm[p], be = nrm[q], ga = s_gam[slot];
                    int rot = 0;
                    const double big = fmax(al, be);
                    if (ga != 0.0 && big > 0.0) {
                        // scale by a power of two so the test and the FP32 ratio cannot over/underflow
                        const int e = ilogb(big);
                        const double as = scalbn(al, -e), bs = scalbn(be, -e), gs = scalbn(ga, -e);
                        if (gs * gs > tol2 * as * bs) {
                            // zeta = (beta - alpha) / (2 gamma): the difference in FP64 (it may cancel),
                            // the ratio and t in FP32 (relative accuracy 1e-7 keeps the convergence
                            // quadratic); c = 1/sqrt(1 + t^2), s = c t in FP64 so that c^2 + s^2 = 1
                            // to FP64 rounding and the rotation stays orthogonal
                            const float zf = (float)(bs - as) / (2.0f * (float)gs);
                            const float az = fabsf(zf);
                            const float tf = az > 1e18f ? 0.5f / zf
                                                        : copysignf(1.0f, zf) / (az + sqrtf(fmaf(az, az, 1.0f)));
                            const double t = (double)tf;
                            const double c = rsqrt(fma(t, t, 1.0));
                            s_c[slot] = c;
                            s_s[slot] = c * t;
                            nrm[p] = fma(-t, ga, al);
                            nrm[q] = fma(t, ga, be);
                            rot = 1;
                            s_any = 1;
                        }
                    }
                    s_rot[slot] = rot;
                }
            }
            __syncthreads();
            for (int slot = warp; slot < cnt; slot += wpb) {                     // (C)
                if (!s_rot[slot]) continue;
                const int pi = base + slot;
                const int a = rr_player(pi, rnd, npad), bq = rr_player(npad - 1 - pi, rnd, npad);
                const int p = min(a, bq), q = max(a, bq);
                const double c = s_c[slot], sn = s_s[slot];
                double* gp = G + (int64_t)p * n;
                double* gq = G + (int64_t)q * n;
                for (int r = lane; r < n; r += 32) {
                    const double x = gp[r], y = gq[r];
                    gp[r] = fma(c, x, -sn * y);
                    gq[r] = fma(sn, x, c * y);
                }
                if (V != nullptr) {
                    double* vp = V + (int64_t)p * npad;
                    double* vq = V + (int64_t)q * npad;
                    for (int r = lane; r < npad; r += 32) {
                        const double x = vp[r], y = vq[r];
                        vp[r] = fma(c, x, -sn * y);
                        vq[r] = fma(sn, x, c * y);
                    }
                }
            }
            if (!grid_sync(ctl, max_wait, epoch)) return;
        }
        if (threadIdx.x == 0 && s_any) atomicAdd(&ctl[kCtlRot + sweep], 1u);
        if (!grid_sync(ctl, max_wait, epoch)) return;
        if (vload(&ctl[kCtlRot + sweep]) == 0u) {
            if (blockIdx.x == 0 && threadIdx.x == 0) ctl[kCtlSweeps] = (unsigned)(sweep + 1);
            return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[kCtlSweeps] = (unsigned)kMaxSweeps;
}

// Block variant (right vectors not accumulated): the block one-sided method of
// Hari and Veselic with the rotations of a block pair done on its Gram matrix.
// The npad columns form nblk blocks of W columns; in each round of a
// round-robin over blocks, CTA c owns one pair of blocks (I, J).  It copies their
// 2W columns C into shared memory and forms M = C^T C from them; one warp then
// runs the round's rotations (the W mini-rounds of W disjoint pairs between I
// and J, and in the first round of a sweep the W - 1 mini-rounds inside I and
// inside J) two-sided on M, M <- R^T M R, accumulating Z = R_1 R_2 ...; finally
// C Z replaces the columns.  Each rotation is computed from the same
// alpha = |g_p|^2, beta = |g_q|^2, gamma = g_p.g_q as in the one-sided method
// (M holds exactly the Gram matrix of the rotated columns, to rounding, and a
// rotation's update of M has errors relative to the norms of the columns it
// mixes, so the relative accuracy is that of the one-sided method).  Every column
// pair meets once per sweep, as in a cyclic sweep; the n-length work of a round
// is two small dense products (the Gram matrix and C Z) over all the CTA's
// threads, and the sequential rotations touch only the 2W x 2W matrices of one
// warp, so a sweep costs nblk - 1 grid barriers and about n warp-local
// mini-rounds instead of n CTA-wide ones.
constexpr int kJGThreads = 256;  // threads of the block kernel

// Rotation parameters of one column pair from alpha = |g_p|^2, beta = |g_q|^2 and
// gamma = g_p.g_q (Rutishauser's formulas); false when |gamma| <= tol sqrt(alpha beta).
// FP64: zeta = (beta - alpha) / (2 gamma) with the difference in FP64 (it may cancel),
// the ratio and t in FP32 (relative accuracy 1e-7 keeps the convergence quadratic),
// c = 1/sqrt(1 + t^2) and s = c t in FP64 so that c^2 + s^2 = 1 to FP64 rounding and
// the rotation stays orthogonal.
__device__ inline bool rot_params(double al, double be, double ga, double tol2, double& c, double& sn, double& t) {
    const double big = fmax(al, be);
    if (!(ga != 0.0 && big > 0.0)) return false;
    // scale by a power of two so the test and the FP32 ratio cannot over/underflow
    const int e = ilogb(big);
    const double as = scalbn(al, -e), bs = scalbn(be, -e), gs = scalbn(ga, -e);
    if (!(gs * gs > tol2 * as * bs)) return false;
    const float zf = (float)(bs - as) / (2.0f * (float)gs);
    const float az = fabsf(zf);
    const float tf = az > 1e18f ? 0.5f / zf : copysignf(1.0f, zf) / (az + sqrtf(fmaf(az, az, 1.0f)));
    t = (double)tf;
    c = rsqrt(fma(t, t, 1.0));
    sn = c * t;
    return true;
}
// Column stride (elements) of the block's columns in shared memory: odd, so that
// the same row of different columns falls in different banks.
__host__ __device__ inline int gram_ld(int n) { return n | 1; }

template <int W>
__host__ __device__ constexpr size_t gram_smem(int n) {
    return sizeof(double) * (size_t)(2 * W) * (size_t)gram_ld(n);
}

// M = C^T C for the 2W columns in shared memory (stride ld): the tiles on and
// above the diagonal of TM x TM register tiles (the others mirrored), each tile's
// rows split over S interleaved lane slices that a shuffle tree sums in a fixed
// order.  A diagonal tile is symmetric bit for bit (x_a x_b = x_b x_a in every fma).
template <int W>
__device__ inline void gram_form(const double* cols, int n, int ld, double (*M)[2 * W + 1]) {
    constexpr int W2 = 2 * W;
    constexpr int TM = W2 >= 8 ? 4 : 2;
    constexpr int NTS = W2 / TM;
    constexpr int NT = NTS * (NTS + 1) / 2;
    constexpr int S0 = kJGThreads / NT;
    constexpr int S = S0 >= 32 ? 32 : (S0 >= 16 ? 16 : (S0 >= 8 ? 8 : (S0 >= 4 ? 4 : (S0 >= 2 ? 2 : 1))));
    static_assert(NT * S <= kJGThreads, "Gram tiling exceeds the block");
    const int t = threadIdx.x;
    int u = t / S;
    const int s = t % S;
    // lanes of one warp share their tile group: a warp is wholly in or out when S
    // divides 32; with S < 32 the last warp may be partly idle, so idle lanes run the
    // loop on tile 0 and drop their sums (the shuffles need every lane)
    const bool live = u < NT;
    if (!live) u = 0;
    if ((t & ~31) >= NT * S) return;  // whole idle warps
    int ti = 0;
    while (u >= NTS - ti) {
        u -= NTS - ti;
        ++ti;
    }
    const int tj = ti + u;
    double acc[TM][TM];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TM; ++b) acc[a][b] = 0.0;
    const double* ca = cols + (size_t)(ti * TM) * ld;
    const double* cb = cols + (size_t)(tj * TM) * ld;
    for (int r = s; r < n; r += S) {
        double x[TM], y[TM];
#pragma unroll
        for (int a = 0; a < TM; ++a) {
            x[a] = ca[(size_t)a * ld + r];
            y[a] = cb[(size_t)a * ld + r];
        }
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int b = 0; b < TM; ++b) acc[a][b] = fma(x[a], y[b], acc[a][b]);
    }
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TM; ++b) {
            double v = acc[a][b];
#pragma unroll
            for (int d = S / 2; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
            if (s == 0 && live) {
                M[ti * TM + a][tj * TM + b] = v;
                M[tj * TM + b][ti * TM + a] = v;
            }
        }
}

// Row stride of Z: 16-byte rows, so that the C Z products read a row of Z two doubles at a time.
template <int W>
__host__ __device__ constexpr int gram_zs() {
    return 2 * W + 2;
}

// acc[j] += x Z_k[j] for j < W2, Z_k a 16-byte aligned row (vector loads, broadcast
// to the warp).
template <int W2>
__device__ inline void gram_axpy_row(double x, const double* zk, double* acc) {
    static_assert(W2 % 2 == 0, "pairs of columns");
#pragma unroll
    for (int j = 0; j < W2; j += 2) {
        const double2 z = *reinterpret_cast<const double2*>(zk + j);
        acc[j] = fma(x, z.x, acc[j]);
        acc[j + 1] = fma(x, z.y, acc[j + 1]);
    }
}

// One mini-round on the block's Gram matrix by warp 0: npr disjoint pairs
// (pp[k], pq[k]) rotated at once; M <- R^T M R and Z <- Z R.  Returns whether any
// pair rotated (warp-uniform).
template <int W>
__device__ inline bool gram_mini_round(double (*M)[2 * W + 1], double (*Z)[gram_zs<W>()], const int* pp, const int* pq,
                                       int npr,
                                       double tol2, double* s_c, double* s_s, int* s_rot) {
    constexpr int W2 = 2 * W;
    const int lane = threadIdx.x & 31;
    int rot = 0;
    if (lane < npr) {
        const int p = pp[lane], q = pq[lane];
        double c = 1.0, sn = 0.0, t = 0.0;
        rot = rot_params(M[p][p], M[q][q], M[p][q], tol2, c, sn, t) ? 1 : 0;
        s_c[lane] = c;
        s_s[lane] = sn;
        s_rot[lane] = rot;
    }
    const bool any = __any_sync(kFull, rot != 0);
    if (!any) return false;
    __syncwarp();
    if (lane < W2) {  // columns: lane = row of M and of Z
        for (int k = 0; k < npr; ++k) {
            if (!s_rot[k]) continue;
            const int p = pp[k], q = pq[k];
            const double c = s_c[k], sn = s_s[k];
            const double x = M[lane][p], y = M[lane][q];
            M[lane][p] = fma(c, x, -sn * y);
            M[lane][q] = fma(sn, x, c * y);
            const double u = Z[lane][p], v = Z[lane][q];
            Z[lane][p] = fma(c, u, -sn * v);
            Z[lane][q] = fma(sn, u, c * v);
        }
    }
    __syncwarp();
    if (lane < W2) {  // rows: lane = column of M
        for (int k = 0; k < npr; ++k) {
            if (!s_rot[k]) continue;
            const int p = pp[k], q = pq[k];
            const double c = s_c[k], sn = s_s[k];
            const double x = M[p][lane], y = M[q][lane];
            M[p][lane] = fma(c, x, -sn * y);
            M[q][lane] = fma(sn, x, c * y);
        }
    }
    __syncwarp();
    return true;
}

// The W mini-rounds between the blocks (pairs (k, W + (k + mr) mod W)) by warp 0
// with the block's Gram matrix in registers: lane r < 2W holds row r of M and of
// Z, the J half of each row stored cyclically shifted by mr (position k holds
// column W + (k + mr) mod W), so that pair k always meets positions k and k of a
// row and no register is indexed at run time.  A rotation acts on the columns of
// M and Z within each lane, and on the rows of M between lane k and its partner
// lane by shuffles.  M and Z enter and leave in shared memory.  Returns whether
// any pair rotated (warp-uniform).
template <int W>
__device__ inline bool gram_rounds_ij(double (*M)[2 * W + 1], double (*Z)[gram_zs<W>()], double tol2) {
    constexpr int W2 = 2 * W;
    const int lane = threadIdx.x & 31;
    const int r = lane < W2 ? lane : 0;  // lanes past 2W mirror row 0 (their results are dropped)
    double A[W], J[W], ZA[W], ZJ[W];
#pragma unroll
    for (int j = 0; j < W; ++j) {
        A[j] = M[r][j];
        J[j] = M[r][W + j];
        ZA[j] = Z[r][j];
        ZJ[j] = Z[r][W + j];
    }
    bool any = false;
    for (int mr = 0; mr < W; ++mr) {
        // own diagonal entry: column r sits at A[r] (r < W) or at J[(r - W - mr) mod W]
        const int jpos = r < W ? r : (r - W - mr + 2 * W) % W;
        double d = 0.0, g = 0.0;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            if (j == jpos) d = r < W ? A[j] : J[j];
            if (j == r) g = J[j];  // M[k][q_k] for the pair's I lane k = r
        }
        const int partner = r < W ? W + (r + mr) % W : jpos;
        const double dq = __shfl_sync(kFull, d, partner);
        double c = 1.0, sn = 0.0, t = 0.0;
        int rot = 0;
        if (lane < W) rot = rot_params(d, dq, g, tol2, c, sn, t) ? 1 : 0;
        if (!rot) {
            c = 1.0;
            sn = 0.0;
        }
        if (!__any_sync(kFull, rot != 0)) {
            // no pair rotates: only the shift of the J halves
        } else {
            any = true;
            // columns (p, q) = (k, W + (k + mr) mod W) of this lane's rows of M and Z
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const double ck = __shfl_sync(kFull, c, k), sk = __shfl_sync(kFull, sn, k);
                const double x = A[k], y = J[k];
                A[k] = fma(ck, x, -sk * y);
                J[k] = fma(sk, x, ck * y);
                const double u = ZA[k], v = ZJ[k];
                ZA[k] = fma(ck, u, -sk * v);
                ZJ[k] = fma(sk, u, ck * v);
            }
            // rows p and q of M: lane p (r < W) and lane q exchange their rows
            const int pair = r < W ? r : jpos;
            const double cp = __shfl_sync(kFull, c, pair), sp = __shfl_sync(kFull, sn, pair);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const double oa = __shfl_sync(kFull, A[k], partner), oj = __shfl_sync(kFull, J[k], partner);
                if (r < W) {
                    A[k] = fma(cp, A[k], -sp * oa);
                    J[k] = fma(cp, J[k], -sp * oj);
                } else {
                    A[k] = fma(sp, oa, cp * A[k]);
                    J[k] = fma(sp, oj, cp * J[k]);
                }
            }
        }
        // next mini-round: position k of the J halves moves to column W + (k + mr + 1) mod W
        const double j0 = J[0], z0 = ZJ[0];
#pragma unroll
        for (int k = 0; k < W - 1; ++k) {
            J[k] = J[k + 1];
            ZJ[k] = ZJ[k + 1];
        }
        J[W - 1] = j0;
        ZJ[W - 1] = z0;
    }
    __syncwarp();
    if (lane < W2) {
#pragma unroll
        for (int j = 0; j < W; ++j) {
            M[r][j] = A[j];
            M[r][W + j] = J[j];
            Z[r][j] = ZA[j];
            Z[r][W + j] = ZJ[j];
        }
    }
    __syncwarp();
    return any;
}

template <int W>
__global__ void __launch_bounds__(kJGThreads, 1) jacobi_gram_kernel(int n, int npad, double* __restrict__ G,
                                                                 unsigned* ctl, double tol, long long max_wait) {
    constexpr int W2 = 2 * W;
    static_assert(W == 1 || W == 2 || W == 4, "block width");
    extern __shared__ __align__(16) unsigned char jsm_raw[];
    double* cols = reinterpret_cast<double*>(jsm_raw);  // 2W columns, stride ld
    __shared__ double M[W2][W2 + 1];
    __shared__ __align__(16) double Z[W2][gram_zs<W>()];
    __shared__ double s_c[W], s_s[W];
    __shared__ int s_rot[W], s_pp[W], s_pq[W];
    __shared__ int s_any, s_rnd;
    if (vload(&ctl[kCtlNeed]) == 0u) {  // every column pair is orthogonal to tol already
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl[kCtlSweeps] = 1u;
        return;
    }
    const double tol2 = tol * tol;
    unsigned epoch = 0;
    const int ld = gram_ld(n);
    const int nblk = npad / W;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        if (threadIdx.x == 0) s_any = 0;
        for (int rnd = 0; rnd < nblk - 1; ++rnd) {
            const int bi = rr_player(blockIdx.x, rnd, nblk), bj = rr_player(nblk - 1 - blockIdx.x, rnd, nblk);
            for (int r = threadIdx.x; r < n; r += blockDim.x) {  // all 2W loads in flight at once
                double v[W2];
#pragma unroll
                for (int k = 0; k < W2; ++k) v[k] = G[(int64_t)(k < W ? bi * W + k : bj * W + (k - W)) * n + r];
#pragma unroll
                for (int k = 0; k < W2; ++k) cols[(size_t)k * ld + r] = v[k];
            }
            __syncthreads();
            gram_form<W>(cols, n, ld, M);
            __syncthreads();
            if (warp == 0) {
                for (int e = lane; e < W2 * W2; e += 32) Z[e / W2][e % W2] = (e / W2 == e % W2) ? 1.0 : 0.0;
                __syncwarp();
                bool any = false;
                if (rnd == 0) {
                    // rotations inside I and inside J: round-robin on W players, W/2 pairs per block
                    for (int mr = 0; mr < W - 1; ++mr) {
                        if (lane < W) {
                            const int blk = lane / (W / 2), seat = lane % (W / 2);
                            const int a = rr_player(seat, mr, W), b2 = rr_player(W - 1 - seat, mr, W);
                            s_pp[lane] = blk * W + min(a, b2);
                            s_pq[lane] = blk * W + max(a, b2);
                        }
                        __syncwarp();
                        any |= gram_mini_round<W>(M, Z, s_pp, s_pq, W, tol2, s_c, s_s, s_rot);
                        __syncwarp();
                    }
                }
                any |= gram_rounds_ij<W>(M, Z, tol2);  // rotations between I and J
                if (lane == 0) {
                    s_rnd = any ? 1 : 0;
                    if (any) s_any = 1;
                }
            }
            __syncthreads();
            if (s_rnd) {
                // C Z: thread r computes row r of the 2W rotated columns (2W independent sums)
                for (int r = threadIdx.x; r < n; r += blockDim.x) {
                    double acc[W2];
#pragma unroll
                    for (int j = 0; j < W2; ++j) acc[j] = 0.0;
#pragma unroll 2
                    for (int k = 0; k < W2; ++k) {
                        const double x = cols[(size_t)k * ld + r];
                        gram_axpy_row<W2>(x, Z[k], acc);
                    }
#pragma unroll
                    for (int j = 0; j < W2; ++j) G[(int64_t)(j < W ? bi * W + j : bj * W + (j - W)) * n + r] = acc[j];
                }
            }
            if (!grid_sync(ctl, max_wait, epoch)) return;
        }
        if (threadIdx.x == 0 && s_any) atomicAdd(&ctl[kCtlRot + sweep], 1u);
        if (!grid_sync(ctl, max_wait, epoch)) return;
        if (vload(&ctl[kCtlRot + sweep]) == 0u) {
            if (blockIdx.x == 0 && threadIdx.x == 0) ctl[kCtlSweeps] = (unsigned)(sweep + 1);
            return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[kCtlSweeps] = (unsigned)kMaxSweeps;
}


// ---- FP32 preconditioning sweeps -------------------------------------------------------
// The block method above in FP32 with blocks of 16 columns, its rows shared by a cluster:
// G (n x npad) and V (npad x npad) are row-major, cluster c of the grid owns the round's
// block pair (I, J), and CTA k of a cluster's C keeps the k-th part of the rows of G and V.
// A round: the 32 columns of the CTA's rows to shared memory; the Gram matrix of its rows of G,
// sent to every CTA of the cluster; the sum of the C partial matrices in rank order, so that
// every CTA has the same M bit for bit; the rotations on M and Z, the same in every CTA; its
// rows times Z; a barrier with the CTAs of its rank in the other clusters, the only ones that
// read its rows.
// The rotations of a mini-round (16 disjoint pairs) are one step of all 256 threads: thread
// (k, l) holds the 2 x 2 block of M at the rows of pair k and the columns of pair l, and two
// rows of Z at the columns of pair l; thread (k, k) computes pair k's rotation.  From one
// mini-round to the next, columns q move by one position between lanes and rows q through
// shared memory.
// Bound by the latency of that chain (16 mini-rounds a round, 15 more in a sweep's first) and
// of the round's loads, cluster exchange and barrier: 24,000 clocks a round, 10,400 of them the
// rotations, 3.1 ms at order 512.  One CTA a block pair, with the rotations in the registers of one
// warp, held 16 SMs and took 13.8 ms.
constexpr int kJ32W = 16;          // columns of a block
constexpr int kJ32Ld = 36;         // row stride (floats) of the 32 columns and of Z: float4 rows
constexpr int kJ32LdM = 48;        // of M: consecutive rows half the banks apart
constexpr int kJ32Threads = 256;
constexpr int kJ32Tiles = 36;      // 4 x 4 tiles on and above the diagonal of M
constexpr int kJ32Tri = 16 * kJ32Tiles;
constexpr int kJ32Slices = kJ32Threads / kJ32Tiles;  // row slices of a CTA's Gram matrix
// A sweep whose largest |cos| is below 2e-3 is the last one: it leaves couplings near its square,
// below the rounding of the accumulated V (5e-6 a pair at order 512).
constexpr float kJ32Again = 4e-6f;
// Control words: the error word, then for every rank a barrier count (a 128-byte line each) and
// its own record of the sweeps to repeat.
constexpr int kJ32Count = 32, kJ32Rot = kJ32Count + 8 * 32, kJ32Words = kJ32Rot + 8 * kMaxSweeps;

// Rotation of a pair in FP32; false when |gamma| <= tol sqrt(alpha beta).  With d = beta -
// alpha and g = 2 gamma: t = g / (d + sign(d) sqrt(d^2 + g^2)), c = 1 / sqrt(1 + t^2), s = c t.
// (Values are scaled, so the approximate instructions see normal numbers only.)
__device__ inline float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ inline float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ inline bool rot32(float al, float be, float ga, float tol2, float& c, float& sn) {
    const float big = fmaxf(al, be);
    if (!(ga != 0.0f && big > 0.0f)) return false;
    // by a power of two, so that neither the test nor the root over- or underflows
    const float f = __int_as_float(max((254 << 23) - (__float_as_int(big) & 0x7F800000), 1 << 23));
    const float as = al * f, bs = be * f, gs = ga * f;
    if (!(gs * gs > tol2 * as * bs)) return false;
    const float d = bs - as, g = 2.0f * gs;
    const float h2 = fmaf(d, d, g * g);
    const float h = h2 * rsqrt_approx(h2);
    const float t = g * rcp_approx(d >= 0.0f ? d + h : d - h);
    c = rsqrt_approx(fmaf(t, t, 1.0f));
    sn = c * t;
    return true;
}

enum J32State : int { kJ32Go = 0, kJ32Done = 1, kJ32Fail = 2 };

// The two halves of a cluster barrier (every thread of every CTA; a release and an acquire).
__device__ inline void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ inline void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__host__ __device__ inline size_t j32_smem(int n, int npad, int C) {
    return sizeof(float) * kJ32Ld * (size_t)((n + C - 1) / C + (npad + C - 1) / C);
}

// The 2 x 2 block (a b; c d) between the pairs with rotations R (rows) and S (columns).
__device__ inline void rot_block(float2 R, float2 S, float& a, float& b, float& c, float& d) {
    const float a1 = fmaf(R.x, a, -R.y * c), c1 = fmaf(R.y, a, R.x * c);
    const float b1 = fmaf(R.x, b, -R.y * d), d1 = fmaf(R.y, b, R.x * d);
    a = fmaf(S.x, a1, -S.y * b1), b = fmaf(S.y, a1, S.x * b1);
    c = fmaf(S.x, c1, -S.y * d1), d = fmaf(S.y, c1, S.x * d1);
}
__device__ inline void rot_row(float2 S, float& x, float& y) {
    const float u = fmaf(S.x, x, -S.y * y);
    y = fmaf(S.y, x, S.x * y);
    x = u;
}

template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(kJ32Threads, 2)
    jacobi32_kernel(int n, int npad, float* G, float* V, unsigned* ctl, float tol, long long max_wait) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) float buf[];  // own rows of G, then of V; 32 columns, stride kJ32Ld
    __shared__ __align__(16) float s_part[kJ32Slices][kJ32Tri];  // Gram matrices of row slices (upper tiles)
    __shared__ __align__(16) float s_in[C][kJ32Tri];             // and of the cluster's CTAs
    __shared__ __align__(16) float M[32][kJ32LdM], Z[32][kJ32Ld];
    __shared__ float2 s_cs[kJ32W];
    __shared__ int s_state[C], s_ok;
    float(*s_q)[2][kJ32W][kJ32W] = reinterpret_cast<float(*)[2][kJ32W][kJ32W]>(&s_part[0][0]);  // rows q, twice
    static_assert(4 * kJ32W * kJ32W <= kJ32Slices * kJ32Tri, "the rotations' exchange fits the partial sums");
    const int tid = threadIdx.x;
    if ((int)cl.num_blocks() != C || (int)gridDim.x != C * (npad / (2 * kJ32W))) {  // not the launch it is built for
        if (blockIdx.x == 0 && tid == 0) atomicOr(&ctl[kCtlErr], 1u);
        return;
    }
    const int rank = (int)cl.block_rank(), pair = (int)blockIdx.x / C, nb = (int)gridDim.x / C;
    const int nblk = npad / kJ32W;
    const float tol2 = tol * tol;
    const int g0 = n * rank / C, ng = n * (rank + 1) / C - g0;
    const int v0 = npad * rank / C, nr = ng + npad * (rank + 1) / C - v0;
    const int q4 = 4 * (tid & 7);              // this thread's 4 of the 32 columns in copies and products
    const int k = tid >> 4, l = tid & 15;      // its pairs in the rotations
    const int k1 = (k + 1) & 15, l1 = (l + 1) & 15;
    // its 4 x 4 tile (ti <= tj) and row slice in the Gram matrix
    const int slice = tid / kJ32Tiles;
    int ti = 0, tj = tid % kJ32Tiles;
    while (tj >= 8 - ti) tj -= 8 - ti, ++ti;
    tj += ti;
    int state = kJ32Go, sweeps = kMaxSweeps;
    bool pending = false;  // an arrival at the cluster barrier that has not been waited for
    unsigned epoch = 0;
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        bool again = false;
        for (int rnd = 0; rnd < nblk - 1; ++rnd) {
            const int bi = rr_player(pair, rnd, nblk), bj = rr_player(nblk - 1 - pair, rnd, nblk);
            const int col = q4 < kJ32W ? bi * kJ32W + q4 : bj * kJ32W + q4 - kJ32W;
#pragma unroll 4
            for (int r = tid >> 3; r < nr; r += kJ32Threads / 8) {
                const float* src = r < ng ? G + (int64_t)(g0 + r) * npad : V + (int64_t)(v0 + r - ng) * npad;
                *reinterpret_cast<float4*>(buf + r * kJ32Ld + q4) = __ldcg(reinterpret_cast<const float4*>(src + col));
            }
            __syncthreads();
            if (slice < kJ32Slices) {  // upper tiles of the Gram matrix of the own rows
                float acc[4][4] = {};
#pragma unroll 2
                for (int r = slice; r < ng; r += kJ32Slices) {
                    const float4 x = *reinterpret_cast<const float4*>(buf + r * kJ32Ld + 4 * ti);
                    const float4 y = *reinterpret_cast<const float4*>(buf + r * kJ32Ld + 4 * tj);
                    const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(xa[a], ya[b], acc[a][b]);
                }
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    *reinterpret_cast<float4*>(&s_part[slice][16 * (tid % kJ32Tiles) + 4 * a]) =
                        make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
            }
            __syncthreads();
            // the cluster's CTAs have read what the round before put into s_in and s_state (the
            // barrier that ends a round joins CTAs of different clusters and does not say so)
            if (pending) cluster_wait();
            if (tid < kJ32Tri / 4) {
                float4 t = *reinterpret_cast<const float4*>(&s_part[0][4 * tid]);
#pragma unroll
                for (int p = 1; p < kJ32Slices; ++p) {
                    const float4 v = *reinterpret_cast<const float4*>(&s_part[p][4 * tid]);
                    t.x += v.x, t.y += v.y, t.z += v.z, t.w += v.w;
                }
#pragma unroll
                for (int c = 0; c < C; ++c)
                    *reinterpret_cast<float4*>(cl.map_shared_rank(&s_in[rank][4 * tid], c)) = t;
            } else if (tid < kJ32Tri / 4 + C) {
                *cl.map_shared_rank(&s_state[rank], tid - kJ32Tri / 4) = state;
            }
            cl.sync();
            if (tid < kJ32Tri / 4) {
                float4 t = *reinterpret_cast<const float4*>(&s_in[0][4 * tid]);
#pragma unroll
                for (int c = 1; c < C; ++c) {
                    const float4 v = *reinterpret_cast<const float4*>(&s_in[c][4 * tid]);
                    t.x += v.x, t.y += v.y, t.z += v.z, t.w += v.w;
                }
                // row tid % 4 of tile tid / 4
                int a = 0, b = tid >> 2;
                while (b >= 8 - a) b -= 8 - a, ++a;
                b += a;
                const int row = 4 * a + (tid & 3);
                *reinterpret_cast<float4*>(&M[row][4 * b]) = t;
                if (a != b) {
                    M[4 * b][row] = t.x;
                    M[4 * b + 1][row] = t.y;
                    M[4 * b + 2][row] = t.z;
                    M[4 * b + 3][row] = t.w;
                }
            }
            // A CTA whose barrier timed out, or that saw a last sweep, leaves together with its
            // cluster (every CTA of which reads the same words): no shared memory is written
            // after its CTA has left.
            if (__syncthreads_or(tid < C && s_state[tid] != kJ32Go)) {
                sweeps = sweep;
                pending = false;
                goto out;
            }
            cluster_arrive();  // s_in and s_state have been read
            pending = true;
            bool any = false;
            float zp[2], zq[2];  // rows k and k + 16 of Z at columns p and q of pair l
#pragma unroll
            for (int e = 0; e < 2; ++e) zp[e] = k + 16 * e == l, zq[e] = k + 16 * e == l + 16;
            if (rnd == 0) {  // rotations inside I and J: round-robin on 16 players in each, 8 pairs a block
                for (int e = tid; e < 32 * 32; e += kJ32Threads) Z[e >> 5][e & 31] = (e >> 5) == (e & 31);
                __syncthreads();
                for (int m = 0; m < kJ32W - 1; ++m) {
                    const int ak = rr_player(k & 7, m, kJ32W), bk = rr_player(15 - (k & 7), m, kJ32W);
                    const int al = rr_player(l & 7, m, kJ32W), bl = rr_player(15 - (l & 7), m, kJ32W);
                    const int pk = 2 * (k & 8) + min(ak, bk), qk = 2 * (k & 8) + max(ak, bk);
                    const int pl = 2 * (l & 8) + min(al, bl), ql = 2 * (l & 8) + max(al, bl);
                    float a = M[pk][pl], b = M[pk][ql], c = M[qk][pl], d = M[qk][ql];
                    float x0 = Z[k][pl], y0 = Z[k][ql], x1 = Z[k + 16][pl], y1 = Z[k + 16][ql];
                    int rot = 0;
                    if (k == l) {
                        float cc = 1.0f, sn = 0.0f;
                        if (rot32(a, d, b, tol2, cc, sn)) {
                            rot = 1;
                            again |= b * b > kJ32Again * a * d;
                        }
                        s_cs[k] = make_float2(cc, sn);
                    }
                    if (!__syncthreads_or(rot)) continue;
                    any = true;
                    const float2 R = s_cs[k], S = s_cs[l];
                    rot_block(R, S, a, b, c, d);
                    rot_row(S, x0, y0);
                    rot_row(S, x1, y1);
                    M[pk][pl] = a, M[pk][ql] = b, M[qk][pl] = c, M[qk][ql] = d;
                    Z[k][pl] = x0, Z[k][ql] = y0, Z[k + 16][pl] = x1, Z[k + 16][ql] = y1;
                    __syncthreads();
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) zp[e] = Z[k + 16 * e][l], zq[e] = Z[k + 16 * e][l + 16];
            }
            {  // rotations between I and J: pair k is (k, 16 + (k + m) mod 16)
                float a = M[k][l], b = M[k][l + 16], c = M[k + 16][l], d = M[k + 16][l + 16];
#pragma unroll 2
                for (int m = 0; m < kJ32W; ++m) {
                    int rot = 0;
                    if (k == l) {
                        float cc = 1.0f, sn = 0.0f;
                        if (rot32(a, d, b, tol2, cc, sn)) {
                            rot = 1;
                            again |= b * b > kJ32Again * a * d;
                        }
                        s_cs[k] = make_float2(cc, sn);
                    }
                    if (__syncthreads_or(rot)) {
                        any = true;
                        const float2 R = s_cs[k], S = s_cs[l];
                        rot_block(R, S, a, b, c, d);
                        rot_row(S, zp[0], zq[0]);
                        rot_row(S, zp[1], zq[1]);
                    }
                    s_q[m & 1][0][k][l] = c;
                    s_q[m & 1][1][k][l] = d;
                    const int next = (tid & 16) | l1;  // the lane of pair l + 1
                    b = __shfl_sync(kFull, b, next);
                    zq[0] = __shfl_sync(kFull, zq[0], next);
                    zq[1] = __shfl_sync(kFull, zq[1], next);
                    __syncthreads();
                    c = s_q[m & 1][0][k1][l];
                    d = s_q[m & 1][1][k1][l1];
                }
            }
            if (any) {
#pragma unroll
                for (int e = 0; e < 2; ++e) Z[k + 16 * e][l] = zp[e], Z[k + 16 * e][l + 16] = zq[e];
                __syncthreads();
                for (int r0 = tid >> 3; r0 < nr; r0 += kJ32Threads / 2) {  // four rows share the reads of Z
                    float acc[4][4] = {};
                    const float* x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[u] = buf + min(r0 + u * (kJ32Threads / 8), nr - 1) * kJ32Ld;
#pragma unroll 2
                    for (int kk = 0; kk < 32; kk += 4) {
                        float4 z[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) z[e] = *reinterpret_cast<const float4*>(&Z[kk + e][q4]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float4 v = *reinterpret_cast<const float4*>(x[u] + kk);
                            const float xs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                acc[u][0] = fmaf(xs[e], z[e].x, acc[u][0]);
                                acc[u][1] = fmaf(xs[e], z[e].y, acc[u][1]);
                                acc[u][2] = fmaf(xs[e], z[e].z, acc[u][2]);
                                acc[u][3] = fmaf(xs[e], z[e].w, acc[u][3]);
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int r = r0 + u * (kJ32Threads / 8);
                        if (r >= nr) break;
                        float* dst = r < ng ? G + (int64_t)(g0 + r) * npad : V + (int64_t)(v0 + r - ng) * npad;
                        *reinterpret_cast<float4*>(dst + col) = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
                    }
                }
            }
            if (rnd == nblk - 2 && again) atomicOr(&ctl[kJ32Rot + rank * kMaxSweeps + sweep], 1u);
            // barrier with the CTAs of this rank; bounded as grid_sync is
            __syncthreads();
            ++epoch;
            if (tid == 0) {
                unsigned* cnt = ctl + kJ32Count + 32 * rank;
                arrive_release(cnt);
                const long long t0 = clock64();
                int ok = 1;
                while (load_acquire(cnt) < epoch * (unsigned)nb) {
                    if (clock64() - t0 > max_wait) {
                        atomicOr(&ctl[kCtlErr], 1u);
                        ok = 0;
                        break;
                    }
                }
                s_ok = ok;
            }
            __syncthreads();
            if (!s_ok) state = kJ32Fail;
        }
        if (state == kJ32Go && vload(&ctl[kJ32Rot + rank * kMaxSweeps + sweep]) == 0u) state = kJ32Done;
    }
out:
    if (blockIdx.x == 0 && tid == 0) ctl[kCtlSweeps] = (unsigned)sweeps;
    if (pending) cluster_wait();
    cl.sync();
}

// FP32 copy of B (n x npad row-major, padded columns zero) and V (npad x npad) = I.
__global__ void jacobi_init32_kernel(int n, int npad, const double* __restrict__ B, int64_t ldb,
                                     float* __restrict__ G, float* __restrict__ V) {
    const int64_t tot = (int64_t)npad * n, totv = (int64_t)npad * npad;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot + totv;
         idx += (int64_t)gridDim.x * blockDim.x) {
        if (idx < tot) {
            const int r = (int)(idx / npad), c = (int)(idx % npad);
            G[idx] = c < n ? (float)B[(int64_t)r * ldb + c] : 0.0f;
        } else {
            const int64_t k = idx - tot;
            V[k] = (k / npad == k % npad) ? 1.0f : 0.0f;
        }
    }
}

// V (n x n row-major, FP64) = the leading n x n block of the accumulated FP32
// rotations V32 (the right singular directions of B to FP32 accuracy).  Also hands
// a timeout of the FP32 sweeps to the status words.
__global__ void jacobi_vinit_kernel(int n, int npad, const float* __restrict__ V32, double* __restrict__ V,
                                    const unsigned* ctl32, int* status) {
    const int64_t tot = (int64_t)n * n;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(idx / n), c = (int)(idx % n);
        V[idx] = (double)V32[(int64_t)r * npad + c];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && ctl32[kCtlErr]) atomicOr(&status[kStTimeout], 1);
}

// After the polar iterations: if V^T V (in T) is not the identity to 1e-12, V = I
// (the FP64 sweeps then start from B itself).  Two kernels over all SMs: the check raises
// `bad` (one CTA took 0.2 ms at order 512), the reset acts on it.
__global__ void __launch_bounds__(256) jacobi_vcheck_kernel(int n, const double* __restrict__ Tm, unsigned* bad) {
    bool off = false;
    for (int idx = (int)(blockIdx.x * blockDim.x + threadIdx.x); idx < n * n; idx += (int)(gridDim.x * blockDim.x)) {
        const int i = idx / n, j = idx % n;
        if (!(fabs(Tm[idx] - (i == j ? 1.0 : 0.0)) <= 1e-12)) off = true;
    }
    if (off) atomicOr(bad, 1u);
}
__global__ void __launch_bounds__(256) jacobi_vreset_kernel(int n, const unsigned* bad, double* __restrict__ V) {
    if (*bad == 0u) return;
    for (int idx = (int)(blockIdx.x * blockDim.x + threadIdx.x); idx < n * n; idx += (int)(gridDim.x * blockDim.x))
        V[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

// ---- all column pairs at once -----------------------------------------------------------
// With the columns of Y nearly orthogonal and M = Y^T Y, the rotations of all pairs together
// are Q = I + E + E^2/2 + E^3/8, E skew with the tangents t_pq of the pairs' rotations:
// Q^T Q = I - E^6/64, orthogonal to FP64 rounding while |E|_2 <= 2^-7.8, and a coupling of
// relative size kappa falls to about kappa^2 / gap.  A column far smaller than the others has
// tangents in proportion, so Y + Y (Q - I) keeps its relative accuracy.
// The first two steps, on V, take Q = the polar factor of I + E by Newton-Schulz iterations
// instead (exact for a pair of close singular values apart from the others).  |E|_2 <= 0.95 needs
// six, |E|_2 <= 0.5 four: the three after the first step and four after the second are enough.
// The bound: |E|_2 <= L + S, S = |E_small|_F / sqrt(2) of the tangents up to `small` and L the
// largest row sum of the others (a few close pairs).  Tangents above `all` are left out, if the
// bound fails those above `mid`, else those above `small`, else all; they stay for the sweeps.
struct TanLimits {
    double all, mid, small, norm;
};
constexpr TanLimits kJTanV1{0.7, 0.35, 0.03, 0.95}, kJTanV2{0.45, 0.2, 0.03, 0.5};
constexpr TanLimits kJTanY{4e-3, 2e-3, 0x1p-10, 4.48e-3};

// Block i: row i of E from M (null E: only the test), its sum of squares up to lim.small, its
// sums from there to lim.mid and to lim.all, and `need` if a coupling of the row exceeds tol.
__global__ void __launch_bounds__(128) jacobi_tan_kernel(int n, const double* __restrict__ M, double tol,
                                                         TanLimits lim, double* __restrict__ E,
                                                         double* __restrict__ rows, unsigned* need) {
    __shared__ double red[3][4];
    const int i = blockIdx.x;
    const double tol2 = tol * tol;
    bool over = false;
    double sq = 0.0, mid = 0.0, all = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int p = min(i, j), q = max(i, j);
        double c, sn, t = 0.0;
        const bool rot = p != q && rot_params(M[p * n + p], M[q * n + q], M[p * n + q], tol2, c, sn, t);
        if (rot) over = true;
        if (!rot || fabs(t) > lim.all) t = 0.0;
        if (E) E[i * n + j] = i < j ? t : -t;
        const double v = fabs(t);
        if (v <= lim.small) sq = fma(v, v, sq);
        else all += v;
        if (v > lim.small && v <= lim.mid) mid += v;
    }
    if (need && __syncthreads_or(over) && threadIdx.x == 0) atomicOr(need, 1u);
    if (!E) return;
    sq = warp_sum(sq), mid = warp_sum(mid), all = warp_sum(all);
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[0][warp] = sq, red[1][warp] = mid, red[2][warp] = all;
    __syncthreads();
    if (threadIdx.x < 3) {
        const double* r = red[threadIdx.x];
        rows[threadIdx.x * n + i] = (r[0] + r[1]) + (r[2] + r[3]);
    }
}

// Block i: row i of E without the tangents that the norm bound leaves out; H = E (null: not wanted).
__global__ void __launch_bounds__(128) jacobi_guard_kernel(int n, const double* __restrict__ rows, TanLimits lim,
                                                           double* __restrict__ E, double* __restrict__ H) {
    __shared__ double red[3][4];
    double sq = 0.0, mid = 0.0, all = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        sq += rows[j];
        mid = fmax(mid, rows[n + j]);
        all = fmax(all, rows[2 * n + j]);
    }
    sq = warp_sum(sq);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        mid = fmax(mid, __shfl_xor_sync(kFull, mid, d));
        all = fmax(all, __shfl_xor_sync(kFull, all, d));
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[0][warp] = sq, red[1][warp] = mid, red[2][warp] = all;
    __syncthreads();
    const double S = sqrt(0.5 * ((red[0][0] + red[0][1]) + (red[0][2] + red[0][3])));
    mid = fmax(fmax(red[1][0], red[1][1]), fmax(red[1][2], red[1][3]));
    all = fmax(fmax(red[2][0], red[2][1]), fmax(red[2][2], red[2][3]));
    const double keep = S + all <= lim.norm   ? lim.all
                        : S + mid <= lim.norm ? lim.mid
                        : S <= lim.norm       ? lim.small
                                              : -1.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int idx = (int)blockIdx.x * n + j;
        const double t = E[idx], v = fabs(t) <= keep ? t : 0.0;
        E[idx] = v;
        if (H) H[idx] = v;
    }
}

// sigma_c = |g_c|, one warp a column.
__global__ void __launch_bounds__(256) jacobi_norm_kernel(int n, int npad, const double* __restrict__ G,
                                                          double* __restrict__ nrm, int* status) {
    const int lane = threadIdx.x & 31, c = (int)blockIdx.x * 8 + ((int)threadIdx.x >> 5);
    if (c >= npad) return;
    const double* g = G + (int64_t)c * n;
    double acc = 0.0;
    for (int r = lane; r < n; r += 32) acc = fma(g[r], g[r], acc);
    acc = warp_sum(acc);
    if (lane == 0) {
        nrm[c] = sqrt(acc);
        if (!isfinite(nrm[c])) atomicOr(&status[kStNonfinite], 1);
    }
}

// One CTA (1024 threads): bitonic sort of the column norms by (sigma desc, index asc).
__global__ void __launch_bounds__(1024) jacobi_sort_kernel(int npad, const double* __restrict__ nrm,
                                                           double* __restrict__ sig, int* __restrict__ perm,
                                                           const unsigned* ctl, int* status) {
    __shared__ double sk[TSVD_MAX_SMALL_SVD];
    __shared__ int si[TSVD_MAX_SMALL_SVD];
    for (int c = threadIdx.x; c < npad; c += blockDim.x) {
        sk[c] = nrm[c];
        si[c] = c;
    }
    int P = 1;
    while (P < npad) P <<= 1;
    for (int c = npad + threadIdx.x; c < P; c += blockDim.x) {
        sk[c] = -1.0;
        si[c] = c;
    }
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < P; i += blockDim.x) {
                const int p = (j == (k >> 1)) ? (i ^ (k - 1)) : (i ^ j);
                if (p > i) {
                    // element p should come first if it is larger, or equal with a smaller index
                    const bool swap = sk[p] > sk[i] || (sk[p] == sk[i] && si[p] < si[i]);
                    if (swap) {
                        const double tk = sk[i];
                        sk[i] = sk[p];
                        sk[p] = tk;
                        const int ti = si[i];
                        si[i] = si[p];
                        si[p] = ti;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int c = threadIdx.x; c < npad; c += blockDim.x) {
        sig[c] = sk[c];
        perm[c] = si[c];
    }
    if (threadIdx.x == 0) {
        status[kStSweeps] = (int)ctl[kCtlSweeps];
        if (ctl[kCtlErr]) atomicOr(&status[kStTimeout], 1);
    }
}

// CTA per output column j < n.  With V accumulated: the sign convention and the
// row-major Ubar, Vbar.  Without V: Ubar = G / sigma only (the sign is fixed
// later, together with the Vbar columns recovered from B^T Ubar).
__global__ void __launch_bounds__(128) jacobi_out_kernel(int n, int npad, const double* __restrict__ G,
                                                         const double* __restrict__ V,
                                                         const double* __restrict__ sig, const int* __restrict__ perm,
                                                         double* __restrict__ Ubar, double* __restrict__ sigma,
                                                         double* __restrict__ Vbar) {
    __shared__ double bv[128];
    __shared__ int bi[128];
    const int j = blockIdx.x;
    const int src = perm[j];
    double sgn = 1.0;
    const double* v = V ? V + (int64_t)src * npad : nullptr;
    if (v) {
        double best = -1.0;
        int besti = 0;
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            const double a = fabs(v[r]);
            if (a > best) {
                best = a;
                besti = r;
            }
        }
        bv[threadIdx.x] = best;
        bi[threadIdx.x] = besti;
        __syncthreads();
        for (int d = 64; d > 0; d >>= 1) {
            if (threadIdx.x < d) {
                const double ob = bv[threadIdx.x + d];
                const int oi = bi[threadIdx.x + d];
                if (ob > bv[threadIdx.x] || (ob == bv[threadIdx.x] && oi < bi[threadIdx.x])) {
                    bv[threadIdx.x] = ob;
                    bi[threadIdx.x] = oi;
                }
            }
            __syncthreads();
        }
        sgn = v[bi[0]] < 0.0 ? -1.0 : 1.0;
    }
    const double sj = sig[j];
    const double inv = sj > 0.0 ? 1.0 / sj : 0.0;
    const double* g = G + (int64_t)src * n;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        Ubar[(int64_t)r * n + j] = sgn * (g[r] * inv);
        if (v) Vbar[(int64_t)r * n + j] = sgn * v[r];
    }
    if (threadIdx.x == 0) sigma[j] = sj;
}

// Breakdown, non-finite and timeout words of a private status block OR-ed into the caller's.
__global__ void fold_status_kernel(const int* __restrict__ from, int* __restrict__ to) {
    const int w = threadIdx.x;
    if ((w == kStBreakdown || w == kStNonfinite || w == kStTimeout) && from[w]) atomicOr(&to[w], 1);
}

// Vbar[:, j] (held unscaled as B^T ubar_j) /= sigma_j, then the pair (ubar_j, vbar_j)
// is flipped so the largest-magnitude entry of vbar_j (first on ties) is positive.
__global__ void __launch_bounds__(128) jacobi_vfix_kernel(int n, const double* __restrict__ sigma,
                                                          double* __restrict__ Ubar, double* __restrict__ Vbar) {
    __shared__ double bv[128];
    __shared__ int bi[128];
    const int j = blockIdx.x;
    const double sj = sigma[j];
    const double inv = sj > 0.0 ? 1.0 / sj : 0.0;
    double best = -1.0;
    int besti = 0;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double a = fabs(Vbar[(int64_t)r * n + j] * inv);
        if (a > best) {
            best = a;
            besti = r;
        }
    }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = besti;
    __syncthreads();
    for (int d = 64; d > 0; d >>= 1) {
        if (threadIdx.x < d) {
            const double ob = bv[threadIdx.x + d];
            const int oi = bi[threadIdx.x + d];
            if (ob > bv[threadIdx.x] || (ob == bv[threadIdx.x] && oi < bi[threadIdx.x])) {
                bv[threadIdx.x] = ob;
                bi[threadIdx.x] = oi;
            }
        }
        __syncthreads();
    }
    const double sgn = (Vbar[(int64_t)bi[0] * n + j] * inv) < 0.0 ? -1.0 : 1.0;
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        Vbar[(int64_t)r * n + j] = sgn * (Vbar[(int64_t)r * n + j] * inv);
        Ubar[(int64_t)r * n + j] = sgn * Ubar[(int64_t)r * n + j];
    }
}

}  // namespace

// Block width of the FP64 block-Jacobi kernel for an order-n SVD without V (at most
// one wave of 152 CTAs, each owning a pair of blocks), or 0 when the per-pair kernel
// is used (V accumulated, or n <= 48: its FP64 rotations of all columns by one SM take 3.9 ms at
// order 64, growing as n^3, the block path 1 ms).
static int block_width(int n) {
    if (n <= 48 || n > 1024) return 0;
    int w = 1;
    while ((n + 2 * w - 1) / (2 * w) > 152) w *= 2;  // up to 4
    return w;
}
static int pad_to(int n, int w) { return (n + 2 * w - 1) / (2 * w) * (2 * w); }

// Buffers of one small SVD, carved identically by the sizing and the run.
struct SvdBufs {
    double *G, *V, *nrm, *sig, *part, *rows_n;
    int* perm;
    unsigned *ctl, *ctl32;
    float *G32, *V32;
    double *Vp, *Tm, *Y;  // preconditioner: V, V^T V, B V (n x n row-major)
    void* oz;
    size_t oz_bytes;
};

static SvdBufs carve_svd(Arena& ar, int n, int npad, int nv, bool precond) {
    SvdBufs b{};
    b.G = ar.take<double>((size_t)n * npad);
    b.V = ar.take<double>((size_t)npad * npad);
    b.nrm = ar.take<double>(npad);
    b.sig = ar.take<double>(npad);
    b.perm = ar.take<int>(npad);
    b.ctl = ar.take<unsigned>(kCtlWords);
    b.part = ar.take<double>(std::max(gemm_tn_ws(nullptr, n, n, nv > 0 ? nv : 1, false),
                                      gemm_tn_ws(nullptr, n, n, n, true)) / sizeof(double) + 1);
    if (precond) {
        const int np32 = pad_to(n, kJ32W);
        b.ctl32 = ar.take<unsigned>(kJ32Words);
        b.G32 = ar.take<float>((size_t)n * np32);
        b.V32 = ar.take<float>((size_t)np32 * np32);
        b.Vp = ar.take<double>((size_t)n * n);
        b.Tm = ar.take<double>((size_t)n * n);
        b.Y = ar.take<double>((size_t)n * n);
        b.rows_n = ar.take<double>((size_t)3 * n);
        b.oz_bytes = std::max(std::max(oz_tn_ws(n, n, n, true), oz_nn_ws(n, n, n)), sizeof(double) * n * n);
        b.oz = ar.take<char>(b.oz_bytes);
    }
    return b;
}

size_t small_svd_ws(int n) {
    size_t best = 0;
    for (int nv : {n, n - 1}) {
        if (nv < 0) continue;
        const bool acc = nv == n;
        const int w = acc ? 0 : block_width(n);
        const int npad = w ? pad_to(n, w) : n + (n & 1);
        Arena ar;
        carve_svd(ar, n, npad, n, w > 0);
        // re-orthonormalisation of the computed right vectors (block CGS-QR, blocks of 128)
        const int bw = n < TSVD_MAX_BLOCK ? n : TSVD_MAX_BLOCK;
        ar.take<double>((size_t)n * n);
        ar.take<int>(kStCount);
        ar.take<double>((size_t)(n - bw) * bw);
        ar.take<char>(orth_ws(nullptr, n, n - bw, bw));
        best = std::max(best, ar.off);
    }
    return best;
}

static int jacobi_grid(const tsvd_handle* h, int npairs, int& block) {
    if (npairs <= 32) {  // one CTA, one warp per pair, __syncthreads between rounds
        block = 32 * npairs;
        return 1;
    }
    block = 32 * kJWarps;
    int nb = (npairs + kJWarps - 1) / kJWarps;
    if (nb > h->sm_count) nb = h->sm_count;
    const int min_nb = (npairs + kMaxSlots - 1) / kMaxSlots;
    if (nb < min_nb) nb = min_nb;
    if (nb > h->jacobi_coop_blocks) return 0;
    return nb;
}

// Cooperative launch of the block-Jacobi sweeps on G (n x npad, column-major) with blocks of W
// columns.
template <int W>
static int launch_gram(tsvd_handle* h, int n, int npad, double* G, unsigned* ctl, double tol, cudaStream_t st) {
    const int nb = npad / W / 2;
    const size_t smem = gram_smem<W>(n);
    static thread_local int configured = -1;
    if (configured != h->device) {
        TSVD_TRY_CUDA(cudaFuncSetAttribute(jacobi_gram_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)gram_smem<W>(1024)));
        configured = h->device;
    }
    int per_sm = 0;
    TSVD_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_gram_kernel<W>, kJGThreads, smem));
    if (per_sm * h->sm_count < nb) return TSVD_ERR_UNSUPPORTED;
    int nn = n, np = npad;
    double t = tol;
    long long mw = h->max_wait;
    void* args[] = {(void*)&nn, (void*)&np, (void*)&G, (void*)&ctl, (void*)&t, (void*)&mw};
    h->launches++;
    TSVD_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi_gram_kernel<W>, dim3(nb), dim3(kJGThreads), args,
                                              smem, st));
    return TSVD_OK;
}

static int run_block_sweeps(tsvd_handle* h, int n, int npad, int w, double* G, unsigned* ctl, double tol,
                            cudaStream_t st) {
    switch (w) {
        case 1: return launch_gram<1>(h, n, npad, G, ctl, tol, st);
        case 2: return launch_gram<2>(h, n, npad, G, ctl, tol, st);
        case 4: return launch_gram<4>(h, n, npad, G, ctl, tol, st);
        default: return TSVD_ERR_UNSUPPORTED;
    }
}
// Cooperative launch of the FP32 sweeps with clusters of C CTAs; false if the chip does not hold
// all of them at once.
template <int C>
static int launch_jacobi32(tsvd_handle* h, int n, int npad, float* G, float* V, unsigned* ctl, float tol,
                           cudaStream_t st, bool& fits) {
    const int nb = npad / (2 * kJ32W);
    static thread_local int configured = -1;
    if (configured != h->device) {
        TSVD_TRY_CUDA(cudaFuncSetAttribute(jacobi32_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)j32_smem(1024, 1024, C)));
        configured = h->device;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nb * C));
    cfg.blockDim = dim3(kJ32Threads);
    cfg.dynamicSmemBytes = j32_smem(n, npad, C);
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int fit = 0;
    TSVD_TRY_CUDA(cudaOccupancyMaxActiveClusters(&fit, jacobi32_kernel<C>, &cfg));
    fits = fit >= nb;
    if (!fits) return TSVD_OK;
    long long mw = h->max_wait;
    void* args[] = {(void*)&n, (void*)&npad, (void*)&G, (void*)&V, (void*)&ctl, (void*)&tol, (void*)&mw};
    h->launches++;
    TSVD_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi32_kernel<C>, cfg.gridDim, cfg.blockDim, args,
                                              cfg.dynamicSmemBytes, st));
    return TSVD_OK;
}
static int run_jacobi32(tsvd_handle* h, int n, int npad, float* G, float* V, unsigned* ctl, float tol,
                        cudaStream_t st) {
    bool fits = false;
    if (h->svd_cluster >= 8) TSVD_TRY(launch_jacobi32<8>(h, n, npad, G, V, ctl, tol, st, fits));
    if (!fits && h->svd_cluster >= 4) TSVD_TRY(launch_jacobi32<4>(h, n, npad, G, V, ctl, tol, st, fits));
    if (!fits) TSVD_TRY(launch_jacobi32<2>(h, n, npad, G, V, ctl, tol, st, fits));
    return fits ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

int small_svd(tsvd_handle* h, int n, const double* B, int64_t ldb, double* Ubar, double* sigma, double* Vbar, int nv,
              Arena& ar, int* status, cudaStream_t st, bool deferred, double target) {
    if (n < 1 || n > TSVD_MAX_SMALL_SVD) return TSVD_ERR_UNSUPPORTED;
    if (nv < 0 || nv > n) return TSVD_ERR_INVALID_ARG;
    const bool accumulate = (nv == n);
    const int w = accumulate ? 0 : block_width(n);
    const int npad = w ? pad_to(n, w) : n + (n & 1);
    const SvdBufs bf = carve_svd(ar, n, npad, nv, w > 0);
    if (!ar.fits()) return TSVD_ERR_WORKSPACE;
    double* G = bf.G;
    double* V = bf.V;
    {  // the Jacobi sweeps (the right-vector products below are timed as products)
        ProfScope prof(h, TSVD_K_SVD, 0.0, 0.0, st);
        TSVD_TRY_CUDA(cudaMemsetAsync(bf.ctl, 0, sizeof(unsigned) * kCtlWords, st));
        const int64_t tot = (int64_t)npad * npad;
        const unsigned ib = (unsigned)((tot + 255) / 256 < 4096 ? (tot + 255) / 256 : 4096);
        // Sweep tolerance tau (columns p, q count as orthogonal once |g_p.g_q| <=
        // tau |g_p||g_q|): max(n, 16) eps by default.  Ritz pairs built on the result
        // have residuals of a small multiple of tau sigma_1: couplings below tau are
        // never rotated away, and with thick restart the converged kept Ritz vectors
        // enter B with exactly such couplings (their columns are then not rotated at
        // all, and the last block rows of their singular vectors stay zero).  A caller
        // that needs residuals below 1e3 n eps (or as small as they get, target 0)
        // gets tau = sqrt(n) eps, the level to which a computed coupling (an n-term
        // FP64 dot product) is itself known.
        double tol = (double)(n > 16 ? n : 16) * kEps;
        if (target >= 0.0 && target < 1e3 * tol) tol = std::sqrt((double)(n > 16 ? n : 16)) * kEps;
        double* Vacc = accumulate ? V : nullptr;
        if (w > 0) {
            // (1) FP32 block-Jacobi sweeps on B with the rotations accumulated in V32: the
            //     right singular directions of B, orthogonal to FP32 rounding (so B V has
            //     columns orthogonal to about eps32 sigma_1 / sigma_j, where the right
            //     vectors from the orthogonalised columns of B^T would leave couplings of
            //     eps32 (sigma_1 / sigma_j)^2 and more FP64 sweeps)
            const int np32 = pad_to(n, kJ32W);
            TSVD_TRY_CUDA(cudaMemsetAsync(bf.ctl32, 0, sizeof(unsigned) * kJ32Words, st));
            h->launches += 2;
            jacobi_init32_kernel<<<(unsigned)std::min<int64_t>(4096, ((int64_t)(n + np32) * np32 + 255) / 256), 256, 0,
                                   st>>>(n, np32, B, ldb, bf.G32, bf.V32);
            TSVD_TRY_CUDA(cudaGetLastError());
            const float tol32 = (float)(n > 16 ? n : 16) * 5.9604645e-08f;  // n 2^-24
            TSVD_TRY(run_jacobi32(h, n, np32, bf.G32, bf.V32, bf.ctl32, tol32, st));
            jacobi_vinit_kernel<<<(unsigned)std::min<int64_t>(4096, ((int64_t)n * n + 255) / 256), 256, 0, st>>>(
                n, np32, bf.V32, bf.Vp, bf.ctl32, status);
            TSVD_TRY_CUDA(cudaGetLastError());
            // (2) V orthogonal to FP64 rounding by polar (Newton-Schulz) steps V <- V (3 I - V^T V) / 2
            //     with FP64-accurate tensor-core products.  After the first (orthogonal to 1e-8) and
            //     after three more all pairs are rotated at once, V <- V (I + E) with E from
            //     (B V)^T (B V); after the last four, a check that falls back to V = I if V^T V is not
            //     the identity to 1e-12.
            // (3) Y = B V: the SVD of B V is that of B with the right vectors rotated by V.  Two more
            //     rounds of all rotations at once, on Y (E in Vp, H in V: both free here), take its
            //     couplings to FP64 rounding unless singular values nearly coincide.
            // (4) The test that a sweep would make: the FP64 sweeps run only if it finds a pair.
            // Up to order 256 the products are shorter on the FP64 pipe (15 us each at order 64, 110 us
            // with slices and cut tiles; 29 and 60 us at order 256).
            const bool pipe = n <= 256;
            const auto tn = [&](const double* X) {  // Tm = X^T X
                if (pipe)
                    return gemm_tn<double, double>(h, n, n, n, X, n, X, n, bf.Tm, n, true, bf.part, st, ~size_t(0),
                                                   true) == cudaSuccess
                               ? TSVD_OK
                               : TSVD_ERR_CUDA;
                return oz_gemm_tn(h, n, n, n, X, n, X, n, bf.Tm, n, true, bf.oz, bf.oz_bytes, status, st);
            };
            const auto nn = [&](double alpha, const double* X, int64_t ldx, const double* Mm, double beta, double* Yo) {
                if (pipe) {
                    if (X == Yo || Mm == Yo) {  // in place through a copy
                        double* const cp = static_cast<double*>(bf.oz);
                        if (cudaMemcpyAsync(cp, Yo, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                            return (int)TSVD_ERR_CUDA;
                        if (X == Yo) X = cp;
                        if (Mm == Yo) Mm = cp;
                    }
                    return gemm_nn<double, double, double>(h, n, n, n, alpha, X, ldx, Mm, n, beta, Yo, n, false, st,
                                                           true) == cudaSuccess
                               ? (int)TSVD_OK
                               : (int)TSVD_ERR_CUDA;
                }
                return oz_gemm_nn(h, n, n, n, alpha, X, ldx, Mm, n, beta, Yo, n, false, bf.oz, bf.oz_bytes, status, st);
            };
            const auto tangents = [&](const TanLimits& lim, double* E, double* H, unsigned* need) {
                // (the steps take out couplings below tol too, as a sweep's other rotations would)
                h->launches += E ? 2 : 1;
                jacobi_tan_kernel<<<n, 128, 0, st>>>(n, bf.Tm, E ? 2 * kEps : tol, lim, E, bf.rows_n, need);
                if (E) jacobi_guard_kernel<<<n, 128, 0, st>>>(n, bf.rows_n, lim, E, H);
                return cudaGetLastError();
            };
            double* const H = bf.V;
            for (int itn = 0; itn < 8; ++itn) {
                TSVD_TRY(tn(bf.Vp));
                TSVD_TRY(nn(-0.5, bf.Vp, n, bf.Tm, 1.5, bf.Vp));
                if (itn == 0 || itn == 3) {
                    TSVD_TRY(nn(1.0, B, ldb, bf.Vp, 0.0, bf.Y));
                    TSVD_TRY(tn(bf.Y));
                    TSVD_TRY_CUDA(tangents(itn == 0 ? kJTanV1 : kJTanV2, H, nullptr, nullptr));
                    TSVD_TRY(nn(1.0, bf.Vp, n, H, 1.0, bf.Vp));
                }
            }
            TSVD_TRY(tn(bf.Vp));
            h->launches += 2;
            const unsigned vb = (unsigned)std::min<int64_t>(304, ((int64_t)n * n + 255) / 256);
            jacobi_vcheck_kernel<<<vb, 256, 0, st>>>(n, bf.Tm, bf.ctl32 + kCtlVBad);
            jacobi_vreset_kernel<<<vb, 256, 0, st>>>(n, bf.ctl32 + kCtlVBad, bf.Vp);
            TSVD_TRY_CUDA(cudaGetLastError());
            TSVD_TRY(nn(1.0, B, ldb, bf.Vp, 0.0, bf.Y));
            for (int itn = 0; itn < 2; ++itn) {
                TSVD_TRY(tn(bf.Y));
                TSVD_TRY_CUDA(tangents(kJTanY, bf.Vp, H, nullptr));
                TSVD_TRY(nn(0.125, bf.Vp, n, bf.Vp, 0.5, H));   // H = E / 2 + E^2 / 8
                TSVD_TRY(nn(1.0, bf.Vp, n, H, 1.0, bf.Vp));     // E + E H = Q - I
                TSVD_TRY(nn(1.0, bf.Y, n, bf.Vp, 1.0, bf.Y));
            }
            TSVD_TRY(tn(bf.Y));
            TSVD_TRY_CUDA(tangents(kJTanY, nullptr, nullptr, bf.ctl + kCtlNeed));
            h->launches++;
            jacobi_init_kernel<<<ib, 256, 0, st>>>(n, npad, bf.Y, n, G, V);
            TSVD_TRY_CUDA(cudaGetLastError());
            TSVD_TRY(run_block_sweeps(h, n, npad, w, G, bf.ctl, tol, st));
        } else {
            h->launches++;
            jacobi_init_kernel<<<ib, 256, 0, st>>>(n, npad, B, ldb, G, V);
            TSVD_TRY_CUDA(cudaGetLastError());
            const int npairs = npad / 2;
            int block = 0;
            const int nblocks = jacobi_grid(h, npairs, block);
            if (nblocks < 1) return TSVD_ERR_UNSUPPORTED;
            const int ppb = (npairs + nblocks - 1) / nblocks;
            h->launches++;
            if (nblocks == 1) {
                jacobi_sweep_kernel<<<1, block, 0, st>>>(n, npad, G, Vacc, bf.nrm, bf.ctl, tol, ppb, h->max_wait);
                TSVD_TRY_CUDA(cudaGetLastError());
            } else {
                int nn = n, np = npad, pp = ppb;
                double t = tol;
                double* nrm = bf.nrm;
                unsigned* ctl = bf.ctl;
                long long mw = h->max_wait;
                void* args[] = {(void*)&nn, (void*)&np, (void*)&G, (void*)&Vacc, (void*)&nrm, (void*)&ctl, (void*)&t,
                                (void*)&pp, (void*)&mw};
                TSVD_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi_sweep_kernel, dim3(nblocks), dim3(block),
                                                          args, 0, st));
            }
        }
        h->launches += 3;
        jacobi_norm_kernel<<<(unsigned)((npad + 7) / 8), 256, 0, st>>>(n, npad, G, bf.nrm, status);
        jacobi_sort_kernel<<<1, 1024, 0, st>>>(npad, bf.nrm, bf.sig, bf.perm, bf.ctl, status);
        jacobi_out_kernel<<<n, 128, 0, st>>>(n, npad, G, Vacc, bf.sig, bf.perm, Ubar, sigma, Vbar);
        TSVD_TRY_CUDA(cudaGetLastError());
    }
    if (!accumulate && nv > 0) {
        // right vectors of the leading nv triplets: vbar_j = B^T ubar_j / sigma_j
        TSVD_TRY_CUDA(gemm_tn(h, n, n, nv, B, ldb, Ubar, n, Vbar, n, false, bf.part, st));
        h->launches++;
        jacobi_vfix_kernel<<<nv, 128, 0, st>>>(n, sigma, Ubar, Vbar);
        TSVD_TRY_CUDA(cudaGetLastError());
        // The columns of Ubar are orthonormal to the sweep tolerance tau, those of
        // B^T Ubar Sigma^-1 only to tau sigma_1 / sigma_j: one block CGS-QR (Alg. 3)
        // pass restores orthonormal right vectors (R = I + O(tau sigma_1 / sigma_nv)).
        // It reports to status words of its own, so that it never consumes the caller's
        // pending breakdown flag; deferred: unsynchronised, its breakdown folded into the
        // caller's flag (the caller then redoes its work checked).
        OrthCtx vctx;
        vctx.seed = 0x5eedULL;
        vctx.deferred = deferred;
        double* Rv = ar.take<double>((size_t)nv * nv);
        int* vst = ar.take<int>(kStCount);
        if (!ar.fits()) return TSVD_ERR_WORKSPACE;
        TSVD_TRY_CUDA(cudaMemsetAsync(vst, 0, sizeof(int) * kStCount, st));
        TSVD_TRY(cgs_qr<double>(h, n, nv, nv < TSVD_MAX_BLOCK ? nv : TSVD_MAX_BLOCK, Vbar, n, Rv, vctx, ar, vst, st));
        h->launches++;
        fold_status_kernel<<<1, 32, 0, st>>>(vst, status);
        TSVD_TRY_CUDA(cudaGetLastError());
    }
    return TSVD_OK;
}

// Co-resident CTAs of the cooperative sweep kernel at its multi-CTA block size.
int jacobi_coop_capacity(int device, int sm_count) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_sweep_kernel, 32 * kJWarps, 0) != cudaSuccess)
        return 0;
    (void)device;
    return per_sm * sm_count;
}

}  // namespace tsvd
