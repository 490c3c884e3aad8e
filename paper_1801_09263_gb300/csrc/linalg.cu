// Dense linear algebra of the exchange path: contractions over the grid
// (Gram-type products such as M = dV Psi^T W of Eq. 3, S of Eq. 4 and the
// Loewdin overlap), orbital combinations (W_loc = phi U, xi = W L^{-T},
// K_ACE psi = -xi X), and the small FP64 N x N factorisations (Cholesky of
// -M', triangular inverse, inverse square roots by Newton-Schulz).
#include <algorithm>
#include <cmath>
#include <vector>
#include <cstdlib>
#include <cstdint>
#include <type_traits>

#include "f32x2.cuh"
#include "chunk_sum.cuh"
#include "lace_internal.cuh"

namespace lace {

namespace {

// ------------------------------------------------------------------ gemm_rows
constexpr int GR_BM = 64, GR_BN = 64, GR_BK = 16, GR_THREADS = 256;
// FP32 path: products of one BK step (16 neighbouring grid points) are summed
// in FP32 and then folded into a compensated (Kahan) FP32 accumulator.  Folding
// less often lets tiny tail products fall below half an ulp of a long running
// sum and vanish, which biases Gram matrices of positive terms low (measured:
// -3.6e-8 relative with 128-product runs on localised orbitals).
constexpr int GR_INNER = 1;

template <typename T> __device__ __forceinline__ T opv(T x, bool a) { return a ? (x < T(0) ? -x : x) : x; }

// Partial C over one K-chunk: work[chunk][m][n] = sum_{r in chunk} op(A[m][r]) op(B[n][r]).
// Four consecutive k of row r of X (zero outside the rows or the chunk).
// VEC: one 16-byte load (the caller guarantees ldx, the base and the chunk
// starts are multiples of 4 elements).
template <typename T, bool VEC>
__device__ __forceinline__ void load4_row(const T* __restrict__ X, size_t ldx, int r, int rows, size_t k, size_t k_end,
                                          bool absval, T* v) {
    v[0] = v[1] = v[2] = v[3] = T(0);
    if (r >= rows) return;
    const T* p = X + (size_t)r * ldx + k;
    if constexpr (VEC && sizeof(T) == 4) {
        if (k + 4 <= k_end) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(p));
            v[0] = opv(q.x, absval); v[1] = opv(q.y, absval); v[2] = opv(q.z, absval); v[3] = opv(q.w, absval);
            return;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (k + c < k_end) v[c] = opv(__ldg(p + c), absval);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(GR_THREADS) gemm_rows_kernel(int M, int N, size_t K, const T* __restrict__ A,
                                                                size_t lda, const T* __restrict__ B, size_t ldb,
                                                                bool absval, bool sym, size_t kchunk,
                                                                double* __restrict__ work) {
    // row pitch GR_BM + 4 keeps the 4-wide reads of a row 16-byte aligned
    __shared__ __align__(16) T As[GR_BK][GR_BM + 4];
    __shared__ __align__(16) T Bs[GR_BK][GR_BN + 4];
    if (sym && blockIdx.y < blockIdx.x) return;  // symmetric: upper tiles only
    const int m0 = blockIdx.x * GR_BM, n0 = blockIdx.y * GR_BN;
    const size_t k_begin = (size_t)blockIdx.z * kchunk;
    const size_t k_end = min(K, k_begin + kchunk);
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    T acc[4][4], fold[4][4], comp[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = T(0); fold[i][j] = T(0); comp[i][j] = T(0); }
    // FP32: the same products and sums on packed pairs (columns 2jj, 2jj + 1),
    // one instruction per two lanes, each lane rounded as the scalar one
    f2 acc2[4][2], fold2[4][2], comp2[4][2];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) { acc2[i][jj] = bc2(0.f); fold2[i][jj] = bc2(0.f); comp2[i][jj] = bc2(0.f); }
    }
    int inner = 0;
    // each thread loads 4 consecutive k of one row of the A tile and of the B
    // tile per step; the next step's values are loaded while this one is used
    const int lrow = tid / 4;       // 0..63
    const int lcol = (tid % 4) * 4;  // 0,4,8,12
    T pa[4], pb[4];
    if (k_begin < k_end) {
        load4_row<T, VEC>(A + (size_t)m0 * lda, lda, lrow, M - m0, k_begin + lcol, k_end, absval, pa);
        load4_row<T, VEC>(B + (size_t)n0 * ldb, ldb, lrow, N - n0, k_begin + lcol, k_end, absval, pb);
    }
    for (size_t k0 = k_begin; k0 < k_end; k0 += GR_BK) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            As[lcol + c][lrow] = pa[c];
            Bs[lcol + c][lrow] = pb[c];
        }
        __syncthreads();
        if (k0 + GR_BK < k_end) {
            load4_row<T, VEC>(A + (size_t)m0 * lda, lda, lrow, M - m0, k0 + GR_BK + lcol, k_end, absval, pa);
            load4_row<T, VEC>(B + (size_t)n0 * ldb, ldb, lrow, N - n0, k0 + GR_BK + lcol, k_end, absval, pb);
        }
#pragma unroll
        for (int kk = 0; kk < GR_BK; ++kk) {
            if constexpr (sizeof(T) == 4) {
                const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
                const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
                const f2 b01 = mk2(b4.x, b4.y), b23 = mk2(b4.z, b4.w);
                const float a[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f2 ai = bc2(a[i]);
                    acc2[i][0] = fma2(ai, b01, acc2[i][0]);
                    acc2[i][1] = fma2(ai, b23, acc2[i][1]);
                }
            } else {
                T a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * b[j];
            }
        }
        __syncthreads();
        if constexpr (sizeof(T) == 4) {
            if (++inner == GR_INNER) {
                inner = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const f2 y = acc2[i][jj] - comp2[i][jj];
                        const f2 t = fold2[i][jj] + y;
                        comp2[i][jj] = (t - fold2[i][jj]) - y;
                        fold2[i][jj] = t;
                        acc2[i][jj] = bc2(0.f);
                    }
            }
        }
    }
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                unpk2(acc2[i][jj], acc[i][2 * jj], acc[i][2 * jj + 1]);
                unpk2(fold2[i][jj], fold[i][2 * jj], fold[i][2 * jj + 1]);
                unpk2(comp2[i][jj], comp[i][2 * jj], comp[i][2 * jj + 1]);
            }
    }
    double* out = work + (size_t)blockIdx.z * M * N;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n >= N) continue;
            out[(size_t)m * N + n] = (double)fold[i][j] - (double)comp[i][j] + (double)acc[i][j];
        }
    }
}

// The FP32 Gram of 16-byte aligned rows without |.|: the same 64 x 64 tiles,
// chunks and compensated fold, with the A and B tiles brought in by cp.async
// through a GA_STAGES-deep ring of row-major [row][k] tiles (the loads of
// step t + 2 in flight while step t is computed), thread (tx, ty) owning
// rows ty + 16 i and columns tx + 16 j (a warp's 16-byte reads of 16
// consecutive rows fall on distinct bank groups with the 20-float pitch), and
// the products paired along k on packed FMAs: each accumulator pair holds the
// even- and odd-k sums of one output, added before the fold.
constexpr int GA_BK = 16, GA_STAGES = 3, GA_PITCH = GA_BK + 4;
static_assert(GA_BK == GR_BK, "the chunk length is a multiple of GR_BK");
__global__ void __launch_bounds__(GR_THREADS) gemm_rows_f32_async_kernel(int M, int N, size_t K,
                                                                         const float* __restrict__ A, size_t lda,
                                                                         const float* __restrict__ B, size_t ldb,
                                                                         bool sym, size_t kchunk,
                                                                         double* __restrict__ work) {
    __shared__ __align__(16) float As[GA_STAGES][GR_BM][GA_PITCH];
    __shared__ __align__(16) float Bs[GA_STAGES][GR_BN][GA_PITCH];
    if (sym && blockIdx.y < blockIdx.x) return;  // symmetric: upper tiles only
    const int m0 = blockIdx.x * GR_BM, n0 = blockIdx.y * GR_BN;
    const size_t k_begin = (size_t)blockIdx.z * kchunk;
    const size_t k_end = min(K, k_begin + kchunk);
    const int nsteps = k_begin < k_end ? (int)((k_end - k_begin + GA_BK - 1) / GA_BK) : 0;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const int crow = tid / 4, cq = tid % 4;  // the 16-byte chunk this thread copies per tile
    const unsigned as_s = (unsigned)__cvta_generic_to_shared(&As[0][crow][cq * 4]);
    const unsigned bs_s = (unsigned)__cvta_generic_to_shared(&Bs[0][crow][cq * 4]);
    constexpr unsigned kStageBytes = GR_BM * GA_PITCH * sizeof(float);
    auto issue = [&](int t) {
        if (t < nsteps) {
            const size_t k = k_begin + (size_t)t * GA_BK + cq * 4;
            const unsigned st = (unsigned)(t % GA_STAGES) * kStageBytes;
            int ab = 0, bb = 0;
            const float* pa = A;
            const float* pb = B;
            if (k < k_end) {
                const int bytes = (int)(min((size_t)4, k_end - k) * sizeof(float));
                if (m0 + crow < M) { ab = bytes; pa = A + (size_t)(m0 + crow) * lda + k; }
                if (n0 + crow < N) { bb = bytes; pb = B + (size_t)(n0 + crow) * ldb + k; }
            }
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(as_s + st), "l"(pa), "r"(ab) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(bs_s + st), "l"(pb), "r"(bb) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per step, empty past the end
    };
    f2 acc[4][4];
    float fold[4][4], comp[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = bc2(0.f); fold[i][j] = 0.f; comp[i][j] = 0.f; }
    issue(0);
    issue(1);
    for (int t = 0; t < nsteps; ++t) {
        issue(t + 2);
        asm volatile("cp.async.wait_group 2;" ::: "memory");  // step t's copies have landed
        __syncthreads();
        const int st = t % GA_STAGES;
#pragma unroll
        for (int kq = 0; kq < GA_BK; kq += 4) {
            float4 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(&Bs[st][tx + 16 * j][kq]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 a = *reinterpret_cast<const float4*>(&As[st][ty + 16 * i][kq]);
                const f2 a01 = mk2(a.x, a.y), a23 = mk2(a.z, a.w);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fma2(a01, mk2(b[j].x, b[j].y), acc[i][j]);
                    acc[i][j] = fma2(a23, mk2(b[j].z, b[j].w), acc[i][j]);
                }
            }
        }
        __syncthreads();  // stage t % GA_STAGES is refilled by issue(t + 3)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float e, o;
                unpk2(acc[i][j], e, o);
                const float y = (e + o) - comp[i][j];
                const float s = fold[i][j] + y;
                comp[i][j] = (s - fold[i][j]) - y;
                fold[i][j] = s;
                acc[i][j] = bc2(0.f);
            }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    double* out = work + (size_t)blockIdx.z * M * N;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx + 16 * j;
            if (n < N) out[(size_t)m * N + n] = (double)fold[i][j] - (double)comp[i][j];
        }
    }
}

// The FP64 Gram.  FP64 issues one warp instruction in 16 clocks an SM, so the
// kernel is bound by its FMAs alone and must not spend any on padding: 16 x 16
// tiles (for symmetric products on and above the diagonal only) and the K range
// split so that every SM has work whatever the size.  One warp holds a tile,
// 2 x 4 outputs a lane, the four warps of a CTA take every fourth 16-point step
// of the CTA's K range and add up through shared memory.  8 x 8 outputs on 24^3:
// 1,050 -> 9 us (64 x 64 tiles in 14 K chunks, 98 % padding); 32 x 32 on 48^3:
// 1,100 -> 170 us.
constexpr int GD_T = 16, GD_WARPS = 4, GD_PITCH = GD_T + 2;
__global__ void __launch_bounds__(32 * GD_WARPS) gemm_rows_f64_kernel(int M, int N, size_t K, const double* __restrict__ A,
                                                                      size_t lda, const double* __restrict__ B, size_t ldb,
                                                                      bool absval, bool sym, size_t kchunk,
                                                                      double* __restrict__ work) {
    __shared__ __align__(16) double As[GD_WARPS][GD_T][GD_PITCH], Bs[GD_WARPS][GD_T][GD_PITCH];  // [k][row]
    int bm, bn;
    if (sym) {
        const int nt = (M + GD_T - 1) / GD_T;
        int left = blockIdx.x;
        bm = 0;
        while (left >= nt - bm) {
            left -= nt - bm;
            ++bm;
        }
        bn = bm + left;
    } else {
        const int nt = (N + GD_T - 1) / GD_T;
        bm = blockIdx.x / nt;
        bn = blockIdx.x % nt;
    }
    const int m0 = bm * GD_T, n0 = bn * GD_T;
    const size_t k_begin = (size_t)blockIdx.y * kchunk, k_end = min(K, k_begin + kchunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kk = lane & 15, half = lane >> 4;
    double pa[8], pb[8];
    auto fetch = [&](size_t k0) {
        const size_t k = k0 + kk;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 2 * i + half;
            pa[i] = k < k_end && m0 + r < M ? opv(__ldg(A + (size_t)(m0 + r) * lda + k), absval) : 0.0;
            pb[i] = k < k_end && n0 + r < N ? opv(__ldg(B + (size_t)(n0 + r) * ldb + k), absval) : 0.0;
        }
    };
    double acc[2][4] = {{0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0}};
    const int lr = lane >> 2, lc = (lane & 3) * 4;
    size_t k0 = k_begin + (size_t)warp * GD_T;
    if (k0 < k_end) fetch(k0);
    for (; k0 < k_end; k0 += GD_T * GD_WARPS) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            As[warp][kk][2 * i + half] = pa[i];
            Bs[warp][kk][2 * i + half] = pb[i];
        }
        __syncwarp();
        if (k0 + GD_T * GD_WARPS < k_end) fetch(k0 + GD_T * GD_WARPS);
#pragma unroll
        for (int q = 0; q < GD_T; ++q) {
            const double a0 = As[warp][q][lr], a1 = As[warp][q][lr + 8];
            const double2 b0 = *reinterpret_cast<const double2*>(&Bs[warp][q][lc]);
            const double2 b1 = *reinterpret_cast<const double2*>(&Bs[warp][q][lc + 2]);
            acc[0][0] = fma(a0, b0.x, acc[0][0]);
            acc[0][1] = fma(a0, b0.y, acc[0][1]);
            acc[0][2] = fma(a0, b1.x, acc[0][2]);
            acc[0][3] = fma(a0, b1.y, acc[0][3]);
            acc[1][0] = fma(a1, b0.x, acc[1][0]);
            acc[1][1] = fma(a1, b0.y, acc[1][1]);
            acc[1][2] = fma(a1, b1.x, acc[1][2]);
            acc[1][3] = fma(a1, b1.y, acc[1][3]);
        }
    }
    __syncthreads();
    double* red = &As[0][0][0];  // [warp][16 x 16]
    static_assert(sizeof(As) >= sizeof(double) * GD_WARPS * GD_T * GD_T, "the partial tiles fit where the stages were");
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) red[warp * GD_T * GD_T + (lr + 8 * i) * GD_T + lc + j] = acc[i][j];
    __syncthreads();
    double* out = work + (size_t)blockIdx.y * M * N;
    for (int e = threadIdx.x; e < GD_T * GD_T; e += blockDim.x) {
        const int m = m0 + e / GD_T, n = n0 + e % GD_T;
        if (m < M && n < N)
            out[(size_t)m * N + n] = (red[e] + red[GD_T * GD_T + e]) + (red[2 * GD_T * GD_T + e] + red[3 * GD_T * GD_T + e]);
    }
}

int sm_count() {
    static const int n = [] {
        int dev = 0, nsm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return 152;
        if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 152;
        return nsm;
    }();
    return n;
}

// CTAs of gemm_rows_kernel resident on the device at once (SMs x occupancy).
int gr_resident() {
    static const int r = [] {
        int dev = 0, nsm = 0, occ = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return 456;
        if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 456;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gemm_rows_kernel<float, true>, GR_THREADS, 0) !=
            cudaSuccess)
            return 456;
        return std::max(1, nsm * std::max(1, occ));
    }();
    return r;
}

// K chunks: as many as fill the resident CTA slots once over the computed
// tiles (upper triangle only for a symmetric product), at least 256 of K each
// (16 steps: 16 orbitals on 32^3 54 us in 32 chunks of 1024, 17 us in 128).
size_t n_chunks_for(int M, int N, size_t K, bool sym) {
    const size_t tm = (size_t)(M + GR_BM - 1) / GR_BM, tn = (size_t)(N + GR_BN - 1) / GR_BN;
    const size_t tiles = sym ? tm * (tm + 1) / 2 : tm * tn;
    const size_t want = std::max<size_t>(1, (size_t)gr_resident() / tiles);
    const size_t maxc = (K + 255) / 256;
    return std::max<size_t>(1, std::min(want, maxc));
}

// The FP64 Gram's CTAs an SM (16 warps: four a scheduler) and its K chunks: one
// round of resident CTAs over the tiles, at least 64 points a warp's step.
constexpr int GD_CTAS = 4;
size_t f64_tiles(int M, int N, bool sym) {
    const size_t tm = (size_t)(M + GD_T - 1) / GD_T, tn = (size_t)(N + GD_T - 1) / GD_T;
    return sym ? tm * (tm + 1) / 2 : tm * tn;
}
size_t f64_chunks(int M, int N, size_t K, bool sym) {
    const size_t want = std::max<size_t>(1, (size_t)GD_CTAS * sm_count() / f64_tiles(M, N, sym));
    return std::max<size_t>(1, std::min(want, (K + 255) / 256));
}

// Whether an FP64 Gram takes the 64-wide tiles of gemm_rows_kernel: their operands
// are reused four times as often, 0.81 ms a tile on 48^3 against 0.066 ms a 16-wide one,
// but the padding is theirs.  On 48^3, 64-wide and 16-wide: 128 x 128 3.37 and 4.25 ms, its
// triangle 3.35 and 2.39; 192 x 192 7.30 and 9.57, triangle 4.78 and 5.45; 96 x 96 3.34 and
// 2.39; a single tile does not fill the chip, 64 x 64 1.18 and 1.01.
bool f64_wide(int M, int N, bool sym) {
    const size_t tm = (size_t)(M + GR_BM - 1) / GR_BM, tn = (size_t)(N + GR_BN - 1) / GR_BN;
    const size_t wide = sym ? tm * (tm + 1) / 2 : tm * tn;
    return wide > 1 && 2 * f64_tiles(M, N, sym) > 25 * wide;
}

// ------------------------------------------------------------------ gemm_combine
constexpr int GC_BR = 128, GC_BN = 64, GC_BK = 16, GC_THREADS = 256;

// The FP64 combination: a thread a grid point, 16 outputs of it, so that N is
// padded to 16 at most (bound by its FMAs; 32 outputs of 32 on 48^3: 400 -> 190
// us against 64-wide tiles).
constexpr int GCD_N = 16, GCD_THREADS = 128, GCD_KC = 128;
__global__ void __launch_bounds__(GCD_THREADS) gemm_combine_f64_kernel(int N, size_t K, int Kc, const double* __restrict__ A,
                                                                       size_t lda, const double* __restrict__ Coef, int ldcoef,
                                                                       double beta, double* __restrict__ Out, size_t ldo) {
    __shared__ __align__(16) double Cs[GCD_KC][GCD_N];
    const size_t r = (size_t)blockIdx.x * GCD_THREADS + threadIdx.x;
    const int n0 = blockIdx.y * GCD_N;
    const double* a = A + min(r, K - 1);
    double acc[GCD_N];
#pragma unroll
    for (int j = 0; j < GCD_N; ++j) acc[j] = 0.0;
    for (int k0 = 0; k0 < Kc; k0 += GCD_KC) {
        const int kn = min(GCD_KC, Kc - k0);
        __syncthreads();
        for (int e = threadIdx.x; e < kn * GCD_N; e += GCD_THREADS) {
            const int k = e / GCD_N, j = e % GCD_N;
            Cs[k][j] = n0 + j < N ? __ldg(Coef + (size_t)(k0 + k) * ldcoef + n0 + j) : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kn; ++k) {
            const double v = __ldg(a + (size_t)(k0 + k) * lda);
#pragma unroll
            for (int j = 0; j < GCD_N; j += 2) {
                const double2 c = *reinterpret_cast<const double2*>(&Cs[k][j]);
                acc[j] = fma(v, c.x, acc[j]);
                acc[j + 1] = fma(v, c.y, acc[j + 1]);
            }
        }
    }
    if (r >= K) return;
#pragma unroll
    for (int j = 0; j < GCD_N; ++j) {
        if (n0 + j >= N) break;
        double* o = Out + (size_t)(n0 + j) * ldo + r;
        *o = beta == 0.0 ? acc[j] : beta * *o + acc[j];
    }
}

template <typename T>
__global__ void __launch_bounds__(GC_THREADS) gemm_combine_kernel(int N, size_t K, int Kc, const T* __restrict__ A,
                                                                   size_t lda, const double* __restrict__ Coef,
                                                                   int ldcoef, double beta, T* __restrict__ Out,
                                                                   size_t ldo) {
    __shared__ T As[GC_BK][GC_BR];
    __shared__ T Cs[GC_BK][GC_BN];
    const size_t r0 = (size_t)blockIdx.x * GC_BR;
    const int n0 = blockIdx.y * GC_BN;
    const int tid = threadIdx.x;
    const int tr = tid % 32;  // 4 r each: r = r0 + tr + 32*i
    const int tn = tid / 32;  // 8 n each: n = n0 + tn*8 + j
    T acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = T(0);
    for (int k0 = 0; k0 < Kc; k0 += GC_BK) {
        // A tile: 16 x 128 = 2048 elements, 8 per thread
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int e = tid + c * GC_THREADS;
            const int kk = e / GC_BR, rr = e % GC_BR;
            const int k = k0 + kk;
            const size_t r = r0 + rr;
            As[kk][rr] = (k < Kc && r < K) ? A[(size_t)k * lda + r] : T(0);
        }
        // Coef tile: 16 x 64 = 1024 elements, 4 per thread
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int e = tid + c * GC_THREADS;
            const int kk = e / GC_BN, nn = e % GC_BN;
            const int k = k0 + kk, n = n0 + nn;
            Cs[kk][nn] = (k < Kc && n < N) ? (T)Coef[(size_t)k * ldcoef + n] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GC_BK; ++kk) {
            T a[4], c[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][tr + 32 * i];
#pragma unroll
            for (int j = 0; j < 8; ++j) c[j] = Cs[kk][tn * 8 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] += a[i] * c[j];
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int n = n0 + tn * 8 + j;
        if (n >= N) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t r = r0 + tr + 32 * i;
            if (r >= K) continue;
            T* o = Out + (size_t)n * ldo + r;
            *o = beta == 0.0 ? acc[i][j] : (T)beta * *o + acc[i][j];
        }
    }
}

// ------------------------------------------------------------------ small FP64
constexpr int SG = 16;

// C = alpha op(A) op(B) + beta C, SG x SG outputs a CTA, one a thread.
__global__ void small_gemm_kernel(int M, int N, int K, const double* __restrict__ A, int lda, bool ta,
                                  const double* __restrict__ B, int ldb, bool tb, double alpha, double beta,
                                  double* __restrict__ C, int ldc) {
    __shared__ double As[SG][SG + 1];
    __shared__ double Bs[SG][SG + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int m = blockIdx.y * SG + ty, n = blockIdx.x * SG + tx;
    double acc = 0.0;
    for (int k0 = 0; k0 < K; k0 += SG) {
        {   // As[ty][tx] = op(A)[m][k0+tx]
            const int k = k0 + tx;
            double v = 0.0;
            if (m < M && k < K) v = ta ? A[(size_t)k * lda + m] : A[(size_t)m * lda + k];
            As[ty][tx] = v;
        }
        {   // Bs[ty][tx] = op(B)[k0+ty][n]
            const int k = k0 + ty;
            double v = 0.0;
            if (n < N && k < K) v = tb ? B[(size_t)n * ldb + k] : B[(size_t)k * ldb + n];
            Bs[ty][tx] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < SG; ++kk) acc = fma(As[ty][kk], Bs[kk][tx], acc);
        __syncthreads();
    }
    if (m < M && n < N) {
        double* c = C + (size_t)m * ldc + n;
        *c = alpha * acc + (beta == 0.0 ? 0.0 : beta * *c);
    }
}

// The same product for small grids (FP64 throughput is per SM, ~2 FMAs a
// clock here, so small products need more CTAs), 8 x 8 outputs a CTA: K in panels of
// SGP_K, every load of a panel issued before any is used (one L2 round trip a
// panel instead of one per 8-wide step), and four partial sums a thread to
// shorten the dependent FMA chain.
constexpr int SGP_K = 256;
__global__ void __launch_bounds__(64) small_gemm_staged_f64_kernel(int M, int N, int K, const double* __restrict__ A,
                                                                   int lda, bool ta, const double* __restrict__ B,
                                                                   int ldb, bool tb, double alpha, double beta,
                                                                   double* __restrict__ C, int ldc) {
    __shared__ double As[8][SGP_K + 1];  // op(A)[m0 + r][k0 + k]
    __shared__ double Bs[SGP_K][8];      // op(B)[k0 + k][n0 + c]
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * 8 + tx;
    const int m0 = blockIdx.y * 8, n0 = blockIdx.x * 8;
    const int m = m0 + ty, n = n0 + tx;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k0 = 0; k0 < K; k0 += SGP_K) {
        const int kp = min(SGP_K, K - k0);
        for (int q = t; q < 8 * kp; q += 64) {
            // A: ta reads along m (consecutive q -> consecutive r), else along k
            const int r = ta ? q % 8 : q / kp, k = ta ? q / 8 : q % kp;
            const int mm = m0 + r, kk = k0 + k;
            As[r][k] = mm < M ? (ta ? A[(size_t)kk * lda + mm] : A[(size_t)mm * lda + kk]) : 0.0;
        }
        for (int q = t; q < 8 * kp; q += 64) {
            const int c = tb ? q / kp : q % 8, k = tb ? q % kp : q / 8;
            const int nn = n0 + c, kk = k0 + k;
            Bs[k][c] = nn < N ? (tb ? B[(size_t)nn * ldb + kk] : B[(size_t)kk * ldb + nn]) : 0.0;
        }
        __syncthreads();
        int k = 0;
        for (; k + 4 <= kp; k += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = fma(As[ty][k + u], Bs[k + u][tx], acc[u]);
        }
        for (; k < kp; ++k) acc[0] = fma(As[ty][k], Bs[k][tx], acc[0]);
        __syncthreads();
    }
    if (m < M && n < N) {
        double* c = C + (size_t)m * ldc + n;
        const double v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
        *c = alpha * v + (beta == 0.0 ? 0.0 : beta * *c);
    }
}

// y = b y + x
__global__ void axpby_kernel(int n, const double* x, double b, double* y) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) y[idx] = fma(b, y[idx], x[idx]);
}

// ------------------------------------------------------------------ Cholesky
constexpr int CH_NB = 32;
static_assert(CH_NB == 32, "the block kernels map one block row or column to the lanes of a warp");

// FP64 runs at ~2 FMAs per clock per SM on this GPU (1/64 of FP32), so the
// factorisation kernels below keep FP64 operations off their serial chains
// (reciprocal square roots and products instead of square roots and
// divisions) and spread independent rows over many SMs.

// Unblocked Cholesky of the diagonal block at k0 (nb x nb) in shared memory,
// thread (r, c) of a 32 x 32 block owning element (r, c).  Per column j:
// warp 0 scales column j by the pivot's reciprocal square root (lane 0 takes
// it), then the threads of the trailing triangle (r >= c > j) do one FMA each.
__global__ void __launch_bounds__(CH_NB * CH_NB) potrf_diag_kernel(int N, double* A, int lda, int k0, int nb,
                                                                   int* flag) {
    __shared__ double D[CH_NB][CH_NB + 1];
    __shared__ double Lc[CH_NB];
    const int tid = threadIdx.x, r = tid / CH_NB, c = tid % CH_NB;
    if (r < nb && c < nb) D[r][c] = A[(size_t)(k0 + r) * lda + k0 + c];
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        if (tid < 32) {
            double ri = 0.0;
            if (tid == 0) {
                double d = D[j][j];
                if (!(d > 0.0)) {
                    atomicExch(flag, 1);
                    d = 1.0;
                }
                ri = rsqrt(d);
            }
            ri = __shfl_sync(0xffffffffu, ri, 0);
            if (tid >= j && tid < nb) {
                const double l = D[tid][j] * ri;  // L_jj = d / sqrt(d) for tid == j
                Lc[tid] = l;
                D[tid][j] = l;
            }
        }
        __syncthreads();
        if (r < nb && c > j && c <= r) D[r][c] = fma(-Lc[r], Lc[c], D[r][c]);
        __syncthreads();
    }
    if (r < nb && c < nb) A[(size_t)(k0 + r) * lda + k0 + c] = (c <= r) ? D[r][c] : 0.0;
}

// Forward substitution across the lanes of one warp: lane l holds s_l of the
// right-hand side on entry and x_l of L x = s on exit (lanes >= nb idle), L
// the lower-triangular block in D with reciprocal diagonal dinv; steps from
// j0 (the lanes below j0 must hold zeros).  At step j, x_j = s_j / L_jj
// reaches every lane by a shuffle and lanes l > j subtract L_lj x_j.
__device__ __forceinline__ double warp_forward_subst(double s, const double (*D)[CH_NB + 1], const double* dinv,
                                                     int nb, int j0) {
    const int lane = threadIdx.x & 31;
    for (int j = j0; j < nb; ++j) {
        const double x = __shfl_sync(0xffffffffu, s, j) * dinv[j];
        if (lane == j) s = x;
        else if (lane > j && lane < nb) s = fma(-D[lane][j], x, s);
    }
    return s;
}

// Rows below the diagonal block: L_ik = A_ik L_kk^{-T}, i.e. L_kk x = a for
// each row a, one warp per row, four rows per CTA.
__global__ void __launch_bounds__(128) trsm_panel_kernel(int N, double* A, int lda, int k0, int nb) {
    __shared__ double D[CH_NB][CH_NB + 1];
    __shared__ double dinv[CH_NB];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) D[e / nb][e % nb] = A[(size_t)(k0 + e / nb) * lda + k0 + e % nb];
    __syncthreads();
    if (threadIdx.x < nb) dinv[threadIdx.x] = 1.0 / D[threadIdx.x][threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int i = k0 + nb + blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (i >= N) return;  // whole warps
    double* row = A + (size_t)i * lda + k0;
    const double s = warp_forward_subst(lane < nb ? row[lane] : 0.0, D, dinv, nb, 0);
    if (lane < nb) row[lane] = s;
}

__global__ void zero_upper_kernel(int N, double* A, int lda) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= N * N) return;
    const int i = idx / N, j = idx % N;
    if (j > i) A[(size_t)i * lda + j] = 0.0;
}

// Inverses of the lower-triangular diagonal blocks, written to X: column c of
// block b solves L x = e_c (one warp per column, four columns per CTA, the
// CH_NB / 4 CTAs of a block side by side).
__global__ void __launch_bounds__(128) trtri_diag_kernel(int N, const double* L, int ldl, double* X, int ldx) {
    constexpr int CPB = CH_NB / 4;  // CTAs per diagonal block
    const int k0 = (blockIdx.x / CPB) * CH_NB;
    const int nb = min(CH_NB, N - k0);
    __shared__ double D[CH_NB][CH_NB + 1];
    __shared__ double dinv[CH_NB];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) D[e / nb][e % nb] = L[(size_t)(k0 + e / nb) * ldl + k0 + e % nb];
    __syncthreads();
    if (threadIdx.x < nb) dinv[threadIdx.x] = 1.0 / D[threadIdx.x][threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int c = (blockIdx.x % CPB) * 4 + (threadIdx.x >> 5);
    if (c >= nb) return;  // whole warps
    const double s = warp_forward_subst(lane == c ? 1.0 : 0.0, D, dinv, nb, c);
    if (lane < nb) X[(size_t)(k0 + lane) * ldx + k0 + c] = lane >= c ? s : 0.0;
}

__global__ void symmetrize_kernel(int N, const double* A, double* B, int mode, double sgn) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= N * N) return;
    const int i = idx / N, j = idx % N;
    double v;
    if (mode == 0) v = 0.5 * (A[(size_t)i * N + j] + A[(size_t)j * N + i]);
    else if (mode == 1) v = (j >= i) ? A[(size_t)i * N + j] : A[(size_t)j * N + i];  // upper kept
    else v = (j <= i) ? A[(size_t)i * N + j] : A[(size_t)j * N + i];                  // lower kept
    B[idx] = sgn * v;
}

__global__ void transpose_kernel(int N, const double* A, double* B) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= N * N) return;
    const int i = idx / N, j = idx % N;
    B[(size_t)j * N + i] = A[idx];
}

template <typename Tin, typename Tout>
__global__ void convert_kernel(const Tin* __restrict__ in, Tout* __restrict__ out, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = (Tout)in[i];
}

// Vector form for 16-byte aligned arrays: 4 elements per thread and
// iteration, two iterations' loads issued together; n4 = n / 4 groups (the
// tail, n % 4 elements, is converted by thread 0 of block 0).
template <typename Tin, typename Tout>
__global__ void convert4_kernel(const Tin* __restrict__ in, Tout* __restrict__ out, size_t n) {
    const size_t n4 = n / 4, stride = (size_t)gridDim.x * blockDim.x;
    auto ld4 = [&](size_t q, Tin* v) {
        if constexpr (sizeof(Tin) == 8) {
            const double2 a = __ldg(reinterpret_cast<const double2*>(in) + 2 * q);
            const double2 b = __ldg(reinterpret_cast<const double2*>(in) + 2 * q + 1);
            v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
        } else {
            const float4 a = __ldg(reinterpret_cast<const float4*>(in) + q);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        }
    };
    auto st4 = [&](size_t q, const Tin* v) {
        if constexpr (sizeof(Tout) == 4) {
            reinterpret_cast<float4*>(out)[q] = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
        } else {
            reinterpret_cast<double2*>(out)[2 * q] = make_double2((double)v[0], (double)v[1]);
            reinterpret_cast<double2*>(out)[2 * q + 1] = make_double2((double)v[2], (double)v[3]);
        }
    };
    size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; q + stride < n4; q += 2 * stride) {
        Tin a[4], b[4];
        ld4(q, a);
        ld4(q + stride, b);
        st4(q, a);
        st4(q + stride, b);
    }
    if (q < n4) {
        Tin a[4];
        ld4(q, a);
        st4(q, a);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (size_t i = 4 * n4; i < n; ++i) out[i] = (Tout)in[i];
}

// FP32 combination with the A tiles double-buffered by cp.async (16-byte
// chunks, zero-filled past the ends) and the coefficient tile one step ahead
// in registers; same tile shape, thread map and summation order as
// gemm_combine_kernel.  Needs lda % 4 == 0 and a 16-byte aligned A.
__global__ void __launch_bounds__(GC_THREADS) gemm_combine_f32_kernel(int N, size_t K, int Kc,
                                                                       const float* __restrict__ A, size_t lda,
                                                                       const double* __restrict__ Coef, int ldcoef,
                                                                       double beta, float* __restrict__ Out,
                                                                       size_t ldo) {
    __shared__ __align__(16) float As[2][GC_BK][GC_BR];
    __shared__ __align__(16) float Cs[2][GC_BK][GC_BN];
    const size_t r0 = (size_t)blockIdx.x * GC_BR;
    const int n0 = blockIdx.y * GC_BN;
    const int tid = threadIdx.x;
    const int tr = tid % 32;  // 4 r each: r = r0 + tr + 32*i
    const int tn = tid / 32;  // 8 n each: n = n0 + tn*8 + j
    // packed accumulators: acc2[i][jj] holds targets 2jj and 2jj + 1 (the
    // same FMAs in the same order as one scalar accumulator per target)
    f2 acc2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) acc2[i][jj] = bc2(0.f);
    const unsigned as_s = (unsigned)__cvta_generic_to_shared(&As[0][0][0]);
    // A tile: 16 rows x 32 chunks of 4 floats, 2 chunks per thread
    auto issue_a = [&](int k0, int buf) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q = tid + c * GC_THREADS;
            const int kk = q / (GC_BR / 4), r4 = 4 * (q % (GC_BR / 4));
            const int k = k0 + kk;
            const size_t r = r0 + r4;
            int bytes = 0;
            const float* src = A;
            if (k < Kc && r < K) {
                bytes = (int)(min((size_t)4, K - r) * 4);
                src = A + (size_t)k * lda + r;
            }
            const unsigned dst = as_s + (unsigned)(((buf * GC_BK + kk) * GC_BR + r4) * 4);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float cr[4];
    auto load_c = [&](int k0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int e = tid + c * GC_THREADS;
            const int kk = e / GC_BN, nn = e % GC_BN;
            const int k = k0 + kk, n = n0 + nn;
            cr[c] = (k < Kc && n < N) ? (float)__ldg(Coef + (size_t)k * ldcoef + n) : 0.f;
        }
    };
    auto store_c = [&](int buf) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int e = tid + c * GC_THREADS;
            Cs[buf][e / GC_BN][e % GC_BN] = cr[c];
        }
    };
    issue_a(0, 0);
    load_c(0);
    store_c(0);
    int buf = 0;
    for (int k0 = 0; k0 < Kc; k0 += GC_BK, buf ^= 1) {
        const bool more = k0 + GC_BK < Kc;
        if (more) {
            issue_a(k0 + GC_BK, buf ^ 1);
            load_c(k0 + GC_BK);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GC_BK; ++kk) {
            float a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[buf][kk][tr + 32 * i];
            const float4 c0 = *reinterpret_cast<const float4*>(&Cs[buf][kk][tn * 8]);
            const float4 c1 = *reinterpret_cast<const float4*>(&Cs[buf][kk][tn * 8 + 4]);
            const f2 cc[4] = {mk2(c0.x, c0.y), mk2(c0.z, c0.w), mk2(c1.x, c1.y), mk2(c1.z, c1.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f2 ai = bc2(a[i]);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) acc2[i][jj] = fma2(ai, cc[jj], acc2[i][jj]);
            }
        }
        if (more) store_c(buf ^ 1);
        __syncthreads();
    }
    float acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) unpk2(acc2[i][jj], acc[i][2 * jj], acc[i][2 * jj + 1]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int n = n0 + tn * 8 + j;
        if (n >= N) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t r = r0 + tr + 32 * i;
            if (r >= K) continue;
            float* o = Out + (size_t)n * ldo + r;
            *o = beta == 0.0 ? acc[i][j] : (float)beta * *o + acc[i][j];
        }
    }
}

__global__ void fill_zero_kernel(double* p, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = 0.0;
}

}  // namespace

// ============================================================================

size_t gemm_rows_work_elems(int M, int N, size_t K) {
    // a symmetric product takes the most chunks; either precision
    return std::max(n_chunks_for(M, N, K, M == N), f64_chunks(M, N, K, M == N)) * (size_t)M * N;
}

template <typename T>
cudaError_t gemm_rows(int M, int N, size_t K, const T* A, size_t lda, const T* B, size_t ldb, double alpha,
                      bool absval, double* C, int ldc, double* work, size_t work_elems, cudaStream_t s,
                      int* launches) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    const bool sym = (A == B) && (lda == ldb) && (M == N);
    const size_t tot = (size_t)M * N;
    if constexpr (sizeof(T) == 8) if (!f64_wide(M, N, sym)) {
        const size_t n = std::min(f64_chunks(M, N, K, sym), work_elems / tot);
        if (n == 0) return cudaErrorInvalidValue;
        size_t kc = (K + n - 1) / n;
        kc = (kc + GD_T - 1) / GD_T * GD_T;
        const size_t nc = (K + kc - 1) / kc;
        gemm_rows_f64_kernel<<<dim3((unsigned)f64_tiles(M, N, sym), (unsigned)nc), 32 * GD_WARPS, 0, s>>>(
            M, N, K, A, lda, B, ldb, absval, sym, kc, work);
        *launches += 2;
        return chunk_sum(M, N, nc, work, alpha, sym, GD_T, C, ldc, s);
    }
    // as many chunks as the workspace holds, up to the balanced count
    const size_t nch = std::min(n_chunks_for(M, N, K, sym), work_elems / ((size_t)M * N));
    if (nch == 0) return cudaErrorInvalidValue;
    size_t kchunk = (K + nch - 1) / nch;
    kchunk = (kchunk + GR_BK - 1) / GR_BK * GR_BK;
    const size_t nch_eff = (K + kchunk - 1) / kchunk;
    dim3 grid((M + GR_BM - 1) / GR_BM, (N + GR_BN - 1) / GR_BN, (unsigned)nch_eff);
    const bool vec = sizeof(T) == 4 && lda % 4 == 0 && ldb % 4 == 0 && ((uintptr_t)A & 15) == 0 &&
                     ((uintptr_t)B & 15) == 0;
    if constexpr (sizeof(T) == 4) {
        if (vec && !absval)
            gemm_rows_f32_async_kernel<<<grid, GR_THREADS, 0, s>>>(M, N, K, A, lda, B, ldb, sym, kchunk, work);
        else if (vec)
            gemm_rows_kernel<T, true><<<grid, GR_THREADS, 0, s>>>(M, N, K, A, lda, B, ldb, absval, sym, kchunk, work);
        else
            gemm_rows_kernel<T, false><<<grid, GR_THREADS, 0, s>>>(M, N, K, A, lda, B, ldb, absval, sym, kchunk, work);
    } else {
        gemm_rows_kernel<T, false><<<grid, GR_THREADS, 0, s>>>(M, N, K, A, lda, B, ldb, absval, sym, kchunk, work);
    }
    *launches += 2;
    return chunk_sum(M, N, nch_eff, work, alpha, sym, GR_BM, C, ldc, s);
}

template <typename T>
cudaError_t gemm_combine(int N, size_t K, int Kc, const T* A, size_t lda, const double* Coef, int ldcoef, double beta,
                         T* Out, size_t ldo, cudaStream_t s, int* launches) {
    if (N <= 0 || K == 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        gemm_combine_f64_kernel<<<dim3((unsigned)((K + GCD_THREADS - 1) / GCD_THREADS), (N + GCD_N - 1) / GCD_N),
                                  GCD_THREADS, 0, s>>>(N, K, Kc, A, lda, Coef, ldcoef, beta, Out, ldo);
        *launches += 1;
        return cudaGetLastError();
    }
    dim3 grid((unsigned)((K + GC_BR - 1) / GC_BR), (N + GC_BN - 1) / GC_BN);
    bool done = false;
    if constexpr (std::is_same<T, float>::value) {
        static const bool off = [] {
            const char* e = getenv("LACE_COMBINE_SYNC");  // tuning: 1 = the synchronous kernel
            return e && e[0] == '1';
        }();
        if (!off && Kc > 0 && lda % 4 == 0 && ((uintptr_t)A & 15) == 0) {
            gemm_combine_f32_kernel<<<grid, GC_THREADS, 0, s>>>(N, K, Kc, A, lda, Coef, ldcoef, beta, Out, ldo);
            done = true;
        }
    }
    if (!done) gemm_combine_kernel<T><<<grid, GC_THREADS, 0, s>>>(N, K, Kc, A, lda, Coef, ldcoef, beta, Out, ldo);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t small_gemm_f64(int M, int N, int K, const double* A, int lda, bool ta, const double* B, int ldb, bool tb,
                           double alpha, double beta, double* C, int ldc, cudaStream_t s, int* launches) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    const dim3 grid((N + SG - 1) / SG, (M + SG - 1) / SG);
    if (grid.x * grid.y < 64) {  // few 16 x 16 tiles (the blocked factorisations): 8 x 8 tiles, K panels staged
        const dim3 g8((N + 7) / 8, (M + 7) / 8);
        small_gemm_staged_f64_kernel<<<g8, dim3(8, 8), 0, s>>>(M, N, K, A, lda, ta, B, ldb, tb, alpha, beta, C, ldc);
    } else {
        small_gemm_kernel<<<grid, dim3(SG, SG), 0, s>>>(M, N, K, A, lda, ta, B, ldb, tb, alpha, beta, C, ldc);
    }
    *launches += 1;
    return cudaGetLastError();
}

// First-order Loewdin correction making F^T G F = I to second order (G =
// identity when G == nullptr): F <- F (3 I - F^T G F) / 2.  F is N x N FP64 (in
// place); work holds 3 N x N.
cudaError_t lowdin_refine(int N, double* F, const double* G, double* work, cudaStream_t s, int* launches) {
    const size_t nn = (size_t)N * N;
    double* GF = work;
    double* E = work + nn;
    double* F2 = work + 2 * nn;
    const double* rhs = F;
    cudaError_t e;
    if (G) {
        if ((e = small_gemm_f64(N, N, N, G, N, false, F, N, false, 1.0, 0.0, GF, N, s, launches))) return e;
        rhs = GF;
    }
    if ((e = small_gemm_f64(N, N, N, F, N, true, rhs, N, false, -0.5, 0.0, E, N, s, launches)) ||
        (e = small_gemm_f64(N, N, N, F, N, false, E, N, false, 1.0, 0.0, F2, N, s, launches)))
        return e;
    axpby_kernel<<<(int)((nn + 255) / 256), 256, 0, s>>>((int)nn, F2, 1.5, F);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t cholesky_lower(int N, double* A, int lda, int* d_flag, int* ok, cudaStream_t s, int* launches) {
    cudaError_t e;
    cudaMemsetAsync(d_flag, 0, sizeof(int), s);
    for (int k0 = 0; k0 < N; k0 += CH_NB) {
        const int nb = std::min(CH_NB, N - k0);
        potrf_diag_kernel<<<1, CH_NB * CH_NB, 0, s>>>(N, A, lda, k0, nb, d_flag);
        *launches += 1;
        const int rem = N - k0 - nb;
        if (rem > 0) {
            trsm_panel_kernel<<<(rem + 3) / 4, 128, 0, s>>>(N, A, lda, k0, nb);
            *launches += 1;
            // A22 -= L21 L21^T
            double* L21 = A + (size_t)(k0 + nb) * lda + k0;
            double* A22 = A + (size_t)(k0 + nb) * lda + k0 + nb;
            if ((e = small_gemm_f64(rem, rem, nb, L21, lda, false, L21, lda, true, -1.0, 1.0, A22, lda, s, launches))) return e;
        }
    }
    zero_upper_kernel<<<(N * N + 255) / 256, 256, 0, s>>>(N, A, lda);
    *launches += 1;
    if ((e = cudaGetLastError()) || !ok) return e;  // !ok: the caller reads d_flag (0 = positive definite)
    int h = 0;
    cudaMemcpyAsync(&h, d_flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    e = cudaStreamSynchronize(s);
    *ok = (h == 0);
    return e;
}

// Blocked L^{-1}: X_ii = L_ii^{-1};  X_ij = -X_ii * sum_{k=j}^{i-1} L_ik X_kj  (j < i).
cudaError_t trtri_lower(int N, const double* L, int ldl, double* X, int ldx, cudaStream_t s, int* launches) {
    cudaMemsetAsync(X, 0, sizeof(double) * (size_t)N * ldx, s);
    const int nblk = (N + CH_NB - 1) / CH_NB;
    trtri_diag_kernel<<<nblk * (CH_NB / 4), 128, 0, s>>>(N, L, ldl, X, ldx);
    *launches += 1;
    // temp rows: use the upper triangle of X?  No: need a separate buffer of nb x N.
    // Work in place: for block row i, compute T = L[i, 0:i] * X[0:i, 0:i] into X[i, 0:i]
    // (X[i, 0:i] is zero before), then X[i, 0:i] = -X_ii * T, using X's
    // unused upper-right area is not safe; so two steps with a small staging
    // area at the end of X's allocation (caller provides ldx*N + CH_NB*N).
    double* stage = X + (size_t)N * ldx;
    cudaError_t e;
    for (int bi = 1; bi < nblk; ++bi) {
        const int i0 = bi * CH_NB;
        const int nb = std::min(CH_NB, N - i0);
        // stage[nb x i0] = L[i0:i0+nb, 0:i0] * X[0:i0, 0:i0]
        e = small_gemm_f64(nb, i0, i0, L + (size_t)i0 * ldl, ldl, false, X, ldx, false, 1.0, 0.0, stage, i0, s, launches);
        if (e) return e;
        // X[i0:i0+nb, 0:i0] = -X_ii * stage
        e = small_gemm_f64(nb, i0, nb, X + (size_t)i0 * ldx + i0, ldx, false, stage, i0, false, -1.0, 0.0,
                           X + (size_t)i0 * ldx, ldx, s, launches);
        if (e) return e;
    }
    return cudaGetLastError();
}

cudaError_t symmetrize(int N, const double* A, double* B, int mode, bool neg, cudaStream_t s, int* launches) {
    symmetrize_kernel<<<(N * N + 255) / 256, 256, 0, s>>>(N, A, B, mode, neg ? -1.0 : 1.0);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t transpose_f64(int N, const double* A, double* B, cudaStream_t s, int* launches) {
    transpose_kernel<<<(N * N + 255) / 256, 256, 0, s>>>(N, A, B);
    *launches += 1;
    return cudaGetLastError();
}

template <typename Tin, typename Tout>
cudaError_t convert(const Tin* in, Tout* out, size_t n, cudaStream_t s, int* launches) {
    if (n == 0) return cudaSuccess;
    if ((((uintptr_t)in | (uintptr_t)out) & 15) == 0 && (std::is_same<Tin, double>::value || std::is_same<Tin, float>::value)) {
        const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>((n / 4 + 255) / 256, 152 * 8));
        convert4_kernel<Tin, Tout><<<blocks, 256, 0, s>>>(in, out, n);
    } else {
        const unsigned blocks = (unsigned)std::min<size_t>((n + 255) / 256, 152 * 16);
        convert_kernel<Tin, Tout><<<blocks, 256, 0, s>>>(in, out, n);
    }
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t fill_zero_f64(double* p, size_t n, cudaStream_t s, int* launches) {
    if (n == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)std::min<size_t>((n + 255) / 256, 152 * 16);
    fill_zero_kernel<<<blocks, 256, 0, s>>>(p, n);
    *launches += 1;
    return cudaGetLastError();
}

template cudaError_t gemm_rows<float>(int, int, size_t, const float*, size_t, const float*, size_t, double, bool,
                                      double*, int, double*, size_t, cudaStream_t, int*);
template cudaError_t gemm_rows<double>(int, int, size_t, const double*, size_t, const double*, size_t, double, bool,
                                       double*, int, double*, size_t, cudaStream_t, int*);
template cudaError_t gemm_combine<float>(int, size_t, int, const float*, size_t, const double*, int, double, float*,
                                         size_t, cudaStream_t, int*);
template cudaError_t gemm_combine<double>(int, size_t, int, const double*, size_t, const double*, int, double, double*,
                                          size_t, cudaStream_t, int*);
template cudaError_t convert<double, float>(const double*, float*, size_t, cudaStream_t, int*);
template cudaError_t convert<float, double>(const float*, double*, size_t, cudaStream_t, int*);
template cudaError_t convert<double, double>(const double*, double*, size_t, cudaStream_t, int*);

}  // namespace lace
