// Tensor-core product for dense A in the mixed-precision form: Y = A X with A
// and X each split into three BF16 pieces (A = A0 + A1 + A2 to 24 significant
// bits, the same for X) and the six cross terms A_i X_j with i + j <= 2
// accumulated in FP32 in tensor memory.  The dropped terms are O(2^-24) relative,
// so the product is as accurate as an FP32 product (the dense products of Alg. 1
// S1/S3 and Alg. 2 S2/S4 in the mixed form, whose accuracy the FP64 final
// Rayleigh-Ritz step relies on).
//
// Kernel structure (sm_103a, one CTA per SM, 320 threads):
//   warp 0     TMA producer: per 64-wide K block, one 3-D box of the three A
//              pieces (128 rows) and one of the three X^T pieces (Npad rows),
//              128-byte swizzled, into a 2-stage ring (96 KB a stage) guarded
//              by mbarriers (boxes 32 wide in 4 stages have twice as many and
//              shorter runs; with the fix-up below 0.56 against 0.545 ms for a
//              20,000^2 x 128 product);
//   warp 1     owns the TMEM allocation (256 columns: two 128 x Npad FP32
//              accumulators) and issues tcgen05.mma (M = 128, N = Npad, K = 16,
//              BF16 x BF16 -> FP32) from one thread, 24 per K block.  Each
//              accumulation covers only kTcChunk K blocks (48 MMAs), alternating
//              between the two accumulators;
//   warps 2-9  epilogue: tcgen05.ld of each finished accumulator (two warps per
//              32 TMEM lanes, half the columns each), added into FP32 registers
//              with round-to-nearest, and the tile part stored to a partial
//              buffer when its K range ends.
// The short accumulations matter: the tensor core's FP32 accumulation does not
// round to nearest, and over the few thousand MMAs of a 20,000-long inner
// dimension its error grew to about 3e-4 of the accumulated value on a
// diagonally dominant matrix (measured), while 48-MMA chunks summed on the CUDA
// cores keep the product at FP32 accuracy.
// Work split: the (tile, K block) iterations are divided evenly over a fixed
// number of CTAs (152: one wave on a GB300) so that every SM gets the same
// share however the tile count falls; a CTA that covers parts of several tiles
// writes one partial tile per part, and a fix-up kernel adds the parts of each
// tile in CTA order (deterministic).
//
// Every mbarrier wait is bounded (clock64); a wait that gives up raises the
// timeout status word, makes the other roles stop, drains the copies and
// products in flight (bounded too) and frees the tensor memory before exit.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "tc_ptx.cuh"
#include "tsvd_internal.cuh"

namespace tsvd {
namespace {

constexpr int kTcM = 128;                          // A rows per tile = TMEM lanes
constexpr int kTcBK = 64;                          // K per stage: 64 BF16 = one 128-byte row
constexpr int kTcRowB = kTcBK * 2;                 // bytes of one tile row
constexpr int kTcStages = 2;
constexpr int kTcPieceA = kTcM * kTcRowB;          // one A piece per stage: 16 KB
constexpr int kTcMaxN = 128;
constexpr int kTcStageBytes = 3 * kTcPieceA + 3 * kTcMaxN * kTcRowB;  // 96 KB
constexpr int kTcSmem = kTcStages * kTcStageBytes + 1024;               // + alignment slack
constexpr int kTcChunk = 2;                         // K blocks per tensor-memory accumulation
constexpr int kTcEpiWarps = 8;                      // two per TMEM lane quarter, half the columns each
constexpr int kTcThreads = 64 + 32 * kTcEpiWarps;
constexpr int kTcWave = 152;
constexpr int kTcTmemCols = 256;
constexpr long long kTcMaxWait = tcx::kMaxWait;

using namespace tcx;

struct TcPlan {
    int64_t tiles, kb, total;  // row tiles, K blocks per tile, tiles x kb
    int ctas, maxseg;
};

__host__ __device__ inline int64_t tc_lo(int64_t c, int64_t total, int G) { return c * total / G; }

// ---- the product kernel ----------------------------------------------------
__global__ void __launch_bounds__(kTcThreads, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmX, int Npad,
                   int64_t KB, int64_t total, int G, int maxseg, float* __restrict__ partial, int* status,
                   long long max_wait) {
    extern __shared__ uint8_t dsm[];
    __shared__ __align__(8) uint64_t bars[2 * kTcStages + 5];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(kTcStages + s); };
    auto accf = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kTcStages + a); };
    auto acce = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kTcStages + 2 + a); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kTcStages + 4);
    volatile int* abort_flag = &s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x;
    const int64_t lo = tc_lo(c, total, G), hi = tc_lo(c + 1, total, G);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kTcStages; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(accf(a), 1);
            mbar_init(acce(a), 32 * kTcEpiWarps);
        }
        mbar_init(drain, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t stage_tx = (uint32_t)(3 * kTcPieceA + 3 * Npad * kTcRowB);

    if (warp == 0) {
        if (elect_one()) {
            // ---- TMA producer
            int64_t it = 0, t = lo / KB, kb = lo - t * KB;
            bool ok = true;
            for (int64_t i = lo; i < hi && ok; ++i, ++it) {
                const int st = (int)(it % kTcStages);
                if (it >= kTcStages) ok = mbar_wait(empty(st), (uint32_t)(((it / kTcStages) - 1) & 1), abort_flag, max_wait);
                if (!ok) break;
                const int kx = (int)(kb * kTcBK);
                const uint32_t sA = base + (uint32_t)st * kTcStageBytes;
                mbar_arrive_expect_tx(full(st), stage_tx);
                tma_load_3d(sA, &tmA, kx, (int)(t * kTcM), 0, full(st));
                tma_load_3d(sA + 3 * kTcPieceA, &tmX, kx, 0, 0, full(st));
                if (++kb == KB) kb = 0, ++t;
            }
            if (!ok) {
                atomicOr(&status[kStTimeout], 1);
                s_abort = 1;
            }
            // copies in flight land before the CTA can exit
            const int64_t first = it > kTcStages ? it - kTcStages : 0;
            for (int64_t j = first; j < it; ++j) {
                const long long t0 = clock64();
                while (!mbar_try_wait(full((int)(j % kTcStages)), (uint32_t)((j / kTcStages) & 1)))
                    if (clock64() - t0 > kTcMaxWait) break;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            // ---- MMA issuer: one accumulation per chunk of kTcChunk K blocks, alternating
            // between the two accumulators so that the epilogue drains one while the
            // other fills
            const uint32_t idesc = idesc_bf16(kTcM, Npad);
            // the six cross terms (A piece, X piece) kept by the split product
            constexpr int kTermA[6] = {0, 0, 1, 0, 1, 2};
            constexpr int kTermX[6] = {0, 1, 0, 2, 1, 0};
            int64_t it = 0, g = 0;  // K blocks and chunks issued by this CTA
            bool ok = true;
            for (int64_t i = lo; i < hi && ok;) {
                const int64_t t = i / KB;
                const int64_t e = min(hi, (t + 1) * KB);
                for (; i < e && ok; ++g) {
                    const int64_t ce = min(e, i + kTcChunk);
                    const int a = (int)(g & 1);
                    if (g >= 2) {
                        ok = mbar_wait(acce(a), (uint32_t)(((g >> 1) - 1) & 1), abort_flag, max_wait);
                        if (!ok) break;
                        fence_after();
                    }
                    const uint32_t d = tmem + (uint32_t)(a * kTcMaxN);
                    uint32_t acc = 0;
                    for (; i < ce; ++i, ++it) {
                        const int st = (int)(it % kTcStages);
                        ok = mbar_wait(full(st), (uint32_t)((it / kTcStages) & 1), abort_flag, max_wait);
                        if (!ok) break;
                        fence_after();
                        const uint32_t sA = base + (uint32_t)st * kTcStageBytes;
                        const uint32_t sX = sA + 3 * kTcPieceA;
#pragma unroll
                        for (int kk = 0; kk < kTcBK / 16; ++kk) {
#pragma unroll
                            for (int tm = 0; tm < 6; ++tm) {
                                const uint64_t ad = sdesc_sw128(sA + (uint32_t)(kTermA[tm] * kTcPieceA + kk * 32));
                                const uint64_t bd =
                                    sdesc_sw128(sX + (uint32_t)(kTermX[tm] * Npad * kTcRowB + kk * 32));
                                mma_bf16(d, ad, bd, idesc, acc);
                                acc = 1;
                            }
                        }
                        commit(empty(st));
                    }
                    if (!ok) break;
                    commit(accf(a));
                }
            }
            if (!ok) {
                atomicOr(&status[kStTimeout], 1);
                s_abort = 1;
            }
            // every product issued has finished before the tensor memory is freed
            commit(drain);
            const long long t0 = clock64();
            while (!mbar_try_wait(drain, 0))
                if (clock64() - t0 > kTcMaxWait) break;
        }
        __syncwarp();
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 and one half of the
        // columns; each chunk's accumulator is added into FP32 registers (round to
        // nearest, unlike the tensor core's accumulation) and each finished tile part
        // is stored as a partial tile
        const int quarter = warp & 3;
        const int half = (warp - 2) >> 2;
        const int ncol = Npad >> 1;  // a multiple of 16
        const int row = quarter * 32 + lane;
        const uint32_t tlane = (uint32_t)(quarter * 32) << 16;
        int64_t g = 0;
        int seg = 0;
        bool ok = true;
        for (int64_t i = lo; i < hi && ok; ++seg) {
            const int64_t t = i / KB;
            const int64_t e = min(hi, (t + 1) * KB);
            float sum[kTcMaxN / 2];
#pragma unroll
            for (int j = 0; j < kTcMaxN / 2; ++j) sum[j] = 0.f;
            for (; i < e; i = min(e, i + kTcChunk), ++g) {
                const int a = (int)(g & 1);
                int w_ok = 1;
                if (lane == 0) w_ok = mbar_wait(accf(a), (uint32_t)((g >> 1) & 1), abort_flag, max_wait) ? 1 : 0;
                w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
                if (!w_ok) {
                    if (lane == 0) {
                        atomicOr(&status[kStTimeout], 1);
                        s_abort = 1;
                    }
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t taddr = tmem + tlane + (uint32_t)(a * kTcMaxN + half * ncol);
#pragma unroll
                for (int c0 = 0; c0 < kTcMaxN / 2; c0 += 16) {
                    if (c0 < ncol) {
                        float v[16];
                        tmem_ld16(taddr + (uint32_t)c0, v);
#pragma unroll
                        for (int q = 0; q < 16; ++q) sum[c0 + q] += v[q];
                    }
                }
                fence_before();
                mbar_arrive(acce(a));
            }
            if (!ok) break;
            float* dst = partial + ((int64_t)(c * maxseg + seg) * kTcM + row) * Npad + half * ncol;
#pragma unroll
            for (int c0 = 0; c0 < kTcMaxN / 2; c0 += 4)
                if (c0 < ncol) reinterpret_cast<float4*>(dst)[c0 / 4] = make_float4(sum[c0], sum[c0 + 1], sum[c0 + 2], sum[c0 + 3]);
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
    }
}

// Y[t*128 + r][col] = sum over the CTAs covering tile t (in CTA order) of their partial tile; a block
// takes 32 rows (a block for 256 elements, each finding its CTAs by 64-bit divisions, took 32 us at
// 20,000 x 128).
constexpr int kTcFixRows = 32;
__global__ void __launch_bounds__(256) tc_fixup_kernel(int64_t M, int w, int Npad, int64_t KB, int64_t total, int G, int maxseg,
                                const float* __restrict__ partial, float* __restrict__ Y, int64_t ldy) {
    __shared__ int s_c0, s_c1;
    const int64_t t = blockIdx.y;
    if (threadIdx.x == 0) {
        auto cta_of = [&](int64_t i) {
            int64_t cc = i * G / total;
            while (cc + 1 < G && tc_lo(cc + 1, total, G) <= i) ++cc;
            while (cc > 0 && tc_lo(cc, total, G) > i) --cc;
            return (int)cc;
        };
        s_c0 = cta_of(t * KB);
        s_c1 = cta_of((t + 1) * KB - 1);
    }
    __syncthreads();
    const int r0 = (int)blockIdx.x * kTcFixRows, rows = (int)min((int64_t)kTcFixRows, M - t * kTcM - r0);
    // the first CTA of the tile may come from an earlier one; the others begin with this tile
    const int64_t first = ((int64_t)s_c0 * maxseg + (t - tc_lo(s_c0, total, G) / KB)) * kTcM;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < rows * w; idx += 256) {
        const int r = r0 + idx / w, col = idx % w;
        float acc = partial[(first + r) * Npad + col];
        for (int cc = s_c0 + 1; cc <= s_c1; ++cc) acc += partial[((int64_t)cc * maxseg * kTcM + r) * Npad + col];
        Y[(t * kTcM + r) * ldy + col] = acc;
    }
}

// Three-way BF16 split: p0 = bf16(v), p1 = bf16(v - p0), p2 = bf16(v - p0 - p1), to 2^-27 of
// v.  An FP64 value enters as v = f + t, f its leading 24 bits and t the other 29 to FP32
// accuracy, taken from the bits: the FP64 pipe (2 instructions a clock and SM) needed 5 ms
// for 20,000^2 entries in either layout.
__device__ inline void split3(float f, float t, __nv_bfloat16& p0, __nv_bfloat16& p1, __nv_bfloat16& p2) {
    p0 = __float2bfloat16_rn(f);
    const float r1 = f - __bfloat162float(p0);  // exact
    p1 = __float2bfloat16_rn(r1 + t);
    const float r2 = r1 - __bfloat162float(p1);  // exact
    p2 = __float2bfloat16_rn(r2 + t);
}
__device__ inline void split3(float v, __nv_bfloat16& p0, __nv_bfloat16& p1, __nv_bfloat16& p2) {
    split3(v, 0.0f, p0, p1, p2);
}
__device__ inline void split3(double v, __nv_bfloat16& p0, __nv_bfloat16& p1, __nv_bfloat16& p2) {
    const uint64_t u = (uint64_t)__double_as_longlong(v);
    const int e = (int)((u >> 52) & 0x7FF) - 1023;  // exponent of a normal value
    if (e >= -74 && e <= 126) {  // 2^(e - 52) is a normal FP32 value too
        const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
        const float f = __uint_as_float(sign | (unsigned)(e + 127) << 23 | ((unsigned)(u >> 29) & 0x7FFFFFu));
        // t = low 29 bits 2^(e - 52), signed
        const float t = (float)((unsigned)u & 0x1FFFFFFFu) * __uint_as_float(sign | (unsigned)(e + 75) << 23);
        split3(f, t, p0, p1, p2);
        return;
    }
    // zeros and values at the ends of the FP32 range
    p0 = __double2bfloat16(v);
    const double r1 = v - (double)__bfloat162float(p0);
    p1 = __double2bfloat16(r1);
    const double r2 = r1 - (double)__bfloat162float(p1);
    p2 = __double2bfloat16(r2);
}

__device__ inline void store_pair(__nv_bfloat16* dst, __nv_bfloat16 a, __nv_bfloat16 b, int pairs, bool second) {
    if (pairs) {
        *reinterpret_cast<__nv_bfloat162*>(dst) = __halves2bfloat162(a, b);
    } else {
        dst[0] = a;
        if (second) dst[1] = b;
    }
}

// Pieces of S (rows x cols, lds) and of its transpose, [3][rows][ld] and [3][cols][ldt] (a
// null output is left out): one read and one split of every entry, tiles of 64 x 64 through
// shared memory, pairs of a row stored together where the output is 4-byte aligned (`pairs`).
// (A pair at an odd end writes one element of the row's padding, which nothing reads: the
// tensor maps stop at the last column.)  One-dimensional grid, column tiles fastest.
template <typename T>
__global__ void __launch_bounds__(256) split3_kernel(int64_t rows, int64_t cols, const T* __restrict__ S, int64_t lds,
                                                     __nv_bfloat16* __restrict__ out, int64_t ld,
                                                     __nv_bfloat16* __restrict__ outt, int64_t ldt, unsigned ct,
                                                     int pairs) {
    __shared__ __nv_bfloat16 tile[3][64][66];
    const int64_t r0 = (int64_t)(blockIdx.x / ct) * 64, c0 = (int64_t)(blockIdx.x % ct) * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
#pragma unroll 4
    for (int r = ty; r < 64; r += 4) {
        const T v = r0 + r < rows && c0 + tx < cols ? S[(r0 + r) * lds + c0 + tx] : T(0);
        split3(v, tile[0][r][tx], tile[1][r][tx], tile[2][r][tx]);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
    for (int u = warp; u < 3 * 64; u += 8) {
        const int p = u >> 6, q = u & 63;
        if (out && r0 + q < rows && c0 + 2 * lane < cols)
            store_pair(out + (p * rows + r0 + q) * ld + c0 + 2 * lane, tile[p][q][2 * lane], tile[p][q][2 * lane + 1],
                       pairs, c0 + 2 * lane + 1 < cols);
        if (outt && c0 + q < cols && r0 + 2 * lane < rows)
            store_pair(outt + (p * cols + c0 + q) * ldt + r0 + 2 * lane, tile[p][2 * lane][q],
                       tile[p][2 * lane + 1][q], pairs, r0 + 2 * lane + 1 < rows);
    }
}

// ---- host side ---------------------------------------------------------------
// 3-D map over pieces [3][rows][ld] (BF16), box 64 (K) x box_rows x 3, 128-byte swizzle.
bool make_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t ld, int box_rows) {
    return make_plane_map(map, base, cols, rows, ld, box_rows, 3);
}

TcPlan tc_plan(int64_t rows, int64_t cols) {
    TcPlan p;
    p.tiles = (rows + kTcM - 1) / kTcM;
    p.kb = std::max<int64_t>(1, (cols + kTcBK - 1) / kTcBK);
    p.total = p.tiles * p.kb;
    p.ctas = (int)std::min<int64_t>(kTcWave, p.total);
    p.maxseg = 1;
    for (int c = 0; c < p.ctas; ++c) {
        const int64_t lo = tc_lo(c, p.total, p.ctas), hi = tc_lo(c + 1, p.total, p.ctas);
        if (hi > lo) p.maxseg = std::max<int>(p.maxseg, (int)((hi - 1) / p.kb - lo / p.kb + 1));
    }
    return p;
}

// N of the MMA: a multiple of 32 so that each epilogue half is a whole number of 16-column loads.
int npad_of(int w) { return std::min(kTcMaxN, (w + 31) / 32 * 32); }

}  // namespace

int64_t bf16x3_ld(int64_t cols) { return (cols + 7) / 8 * 8; }

size_t bf16x3_bytes(int64_t rows, int64_t cols) { return align256((size_t)3 * rows * bf16x3_ld(cols) * 2); }

template <typename T>
cudaError_t bf16x3_split(tsvd_handle* h, int64_t rows, int64_t cols, const T* S, int64_t lds, void* out, void* outt,
                         cudaStream_t st) {
    if (rows == 0 || cols == 0) return cudaSuccess;
    h->launches++;
    const int64_t ct = (cols + 63) / 64;
    const int pairs = ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(outt)) & 3) == 0;
    split3_kernel<T><<<(unsigned)(ct * ((rows + 63) / 64)), 256, 0, st>>>(
        rows, cols, S, lds, static_cast<__nv_bfloat16*>(out), bf16x3_ld(cols), static_cast<__nv_bfloat16*>(outt),
        bf16x3_ld(rows), (unsigned)ct, pairs);
    return cudaGetLastError();
}
template cudaError_t bf16x3_split<double>(tsvd_handle*, int64_t, int64_t, const double*, int64_t, void*, void*,
                                          cudaStream_t);
template cudaError_t bf16x3_split<float>(tsvd_handle*, int64_t, int64_t, const float*, int64_t, void*, void*,
                                         cudaStream_t);

size_t tc_mm_ws(int64_t rows, int64_t cols, int w) {
    const TcPlan p = tc_plan(rows, cols);
    const int np = npad_of(std::max(w, 1));
    return bf16x3_bytes(np, cols) + align256(sizeof(float) * (size_t)p.ctas * p.maxseg * kTcM * np);
}

cudaError_t tc_mm(tsvd_handle* h, int64_t rows, int64_t cols, const void* pieces, int w, const float* X, int64_t ldx,
                  float* Y, int64_t ldy, void* ws, int* status, cudaStream_t st) {
    if (rows == 0 || w == 0) return cudaSuccess;
    if (cols == 0) {
        for (int64_t i = 0; i < rows; ++i) {
            cudaError_t e = cudaMemsetAsync(Y + i * ldy, 0, sizeof(float) * w, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    static thread_local int configured = -1;
    if (configured != h->device) {
        cudaError_t e = cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
        if (e != cudaSuccess) return e;
        configured = h->device;
    }
    const TcPlan p = tc_plan(rows, cols);
    const int64_t lda = bf16x3_ld(cols);
    ProfScope prof(h, TSVD_K_APROD, 2.0 * rows * cols * w, 2.0 * 3 * rows * cols + 4.0 * (cols + rows) * w, st);
    for (int c0 = 0; c0 < w; c0 += kTcMaxN) {
        const int wp = std::min(kTcMaxN, w - c0);
        const int np = npad_of(wp);
        uint8_t* xp = static_cast<uint8_t*>(ws);
        float* part = reinterpret_cast<float*>(xp + bf16x3_bytes(np, cols));
        // X^T pieces: wp x cols (K-major), rows wp..np-1 come from the map's zero fill
        cudaError_t e = bf16x3_split<float>(h, cols, wp, X + c0, ldx, nullptr, xp, st);
        if (e != cudaSuccess) return e;
        CUtensorMap mA, mX;
        if (!make_map(&mA, pieces, cols, rows, lda, kTcM)) return cudaErrorInvalidValue;
        if (!make_map(&mX, xp, cols, wp, bf16x3_ld(cols), np)) return cudaErrorInvalidValue;
        h->launches += 2;
        tc_gemm_kernel<<<p.ctas, kTcThreads, kTcSmem, st>>>(mA, mX, np, p.kb, p.total, p.ctas, p.maxseg, part,
                                                            status, h->max_wait);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const dim3 fg((unsigned)(kTcM / kTcFixRows), (unsigned)p.tiles);
        tc_fixup_kernel<<<fg, 256, 0, st>>>(rows, wp, np, p.kb, p.total, p.ctas, p.maxseg, part, Y + c0, ldy);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace tcx {

EncodeTiledFn encode_fn() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

bool make_plane_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t ld, int box_rows,
                    int planes) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)(ld * rows) * 2};
    const cuuint32_t box[3] = {(cuuint32_t)kTcBK, (cuuint32_t)box_rows, (cuuint32_t)planes};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tcx
}  // namespace tsvd
