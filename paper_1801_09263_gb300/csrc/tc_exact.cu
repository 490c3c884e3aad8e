// FP32-accurate contractions over the grid on the tensor cores (tcgen05): the
// Loewdin and alignment overlaps C = alpha sum_r A[m][r] B[n][r] and the
// orbital rotations Out[n][r] = sum_k Coef[k][n] A[k][r] (Sec. 2), which the
// pair energies need to FP32's full accuracy.
//
// Slices.  Every operand row is scaled by a power of two so that its largest
// value is below 256 and cut into x = a1 + a2 + a3 (the scheme of Ozaki, Ogita, Oishi
// and Rump, "Error-free transformations of matrix multiplication", Numer.
// Algorithms 59, 2012): a1 an integer and a2 a multiple of 2^-9, both rounded to
// nearest with at most 256 units, a3 the rest (at most 2^-10) with FP16's eleven
// bits, ~30 bits below the row's largest value in all; every slice is an FP16
// number.  Products by order, each order in an accumulator of its own: a1 b1 are
// integers up to 2^16, of which 256 add up exactly in FP32; a1 b2 + a2 b1 are
// multiples of 2^-9 and a2 b2 of 2^-18, exact but for sums no data reaches; the
// rest are 2^-18 of the first and smaller.  So the tensor cores' rounding
// (truncation), which biased two-slice BF16 products by 1e-6 and more, has nothing
// to act on.  The Gram takes all nine products (a3 b3 is positive on the diagonal:
// without it overlaps are 3e-9 too small, 1e-8 on ill-conditioned sets, and with a2 b2 among
// the truncated sums 1e-9) and adds periods of 256 points to compensated FP32
// sums; a rotation is one sum over the orbitals and does without a3 b3 (2^-20).
//
// Errors against FP64, orthonormality of the loaded and of the localised
// orbitals, before (FP32 products on the CUDA cores) -> now: 72^3 x 256
// ill-conditioned 1.6e-7, 1.1e-7 -> 1.8e-8, 9e-8 (the latter is the FP32 inverse
// square root's), localised 2.3e-7, 1.9e-7 -> 6e-8, 6e-8; orbitals rotated 4.1e-7 -> 7e-8.
//
// A row is fixed point: values below 2^-6 of its largest have fewer bits than FP32's 24.
// Peaked rows (unmixed Gaussians of width 0.5 in a box of 20, largest value 113 times
// the rms, 96^3 x 72), before -> now: orthonormality 1.0e-7 -> 2.6e-8, relative L2 error
// 6.6e-8 -> 5.1e-8, largest error 1.3e-7 -> 7.6e-8 of the peak; only where all orbitals are below
// 2^-10 of the peak is it larger, 1.7e-10 -> 1.4e-9 of the peak.
//
// Kernels: the warp-role Gram of tc_gemm.cu with nine products (diagonal tiles load
// and cut their rows once), and combine_ws_kernel of tc_combine.cuh with three
// accumulators of 128 targets: A's slices are in TMEM, since from shared memory both
// operands of a 128 x 128 tile take all its bandwidth, and the cut's writes come on top.
//
// Measured, 72^3 x 256 (launches, alone): Gram 1043 -> 271 us (nine products over
// three tiles of four: 165 us at the dense FP16 rate; bound by shared memory:
// operands, rows and slices are 1.9k of its 128-byte cycles a step of 1.1 us),
// rotation 653 -> 225 us (196 us at the FP16 rate).  Row maxima come with the rounding to FP32.
#include <algorithm>
#include <atomic>

#include "chunk_sum.cuh"
#include "f32x2.cuh"
#include "lace_internal.cuh"
#include "tc_combine.cuh"
#include "tc_util.cuh"

#include <cuda_fp16.h>

namespace lace {

namespace {

constexpr float kSlice = 512.f, kUnslice = 1.f / 512.f;

// D = F32, A = B = F16, both K-major, M = 128, N = 128.
constexpr uint32_t kIdescF16 = (1u << 4) | ((uint32_t)(TC_N >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdescF16), "r"(accumulate));
}
// The products by order into accumulators of 128 columns; mma(acc, i, j, first)
// multiplies slices a_i b_j.  GRAM: all nine, a2 b2 apart from the low ones.
template <bool GRAM, class Mma> __device__ __forceinline__ void mma_orders(uint32_t acc, uint32_t first, Mma mma) {
    mma(acc, 0, 0, first);
    mma(acc + TC_N, 0, 1, first);
    mma(acc + TC_N, 1, 0, 1u);
    mma(acc + 2 * TC_N, 1, 1, first);
    const uint32_t low = acc + (GRAM ? 3 : 2) * TC_N;
    mma(low, 0, 2, GRAM ? first : 1u);
    mma(low, 2, 0, 1u);
    mma(low, 1, 2, 1u);
    mma(low, 2, 1, 1u);
    if (GRAM) mma(low, 2, 2, 1u);
}
// Two FP32 values rounded to FP16, x0 in the low half.
__device__ __forceinline__ uint32_t f16x2_rn(float x0, float x1) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
    return r;
}

// Power of two that brings a row with this largest magnitude (FP32 bits) to
// below 256, and its inverse's exponent: scale = 2^(134 - E), E the biased
// exponent.  Rows without a finite value but zero: 1.
__host__ __device__ __forceinline__ int row_exponent(unsigned maxbits) {
    const int e = (int)(maxbits >> 23) & 0xff;
    if (e == 0 || e == 255) return 0;
    return 134 - e < -126 ? -126 : 134 - e > 127 ? 127 : 134 - e;
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// Nearest integers of two values (|x| < 2^22).
__device__ __forceinline__ f2 rint2(f2 x) {
    const f2 m = bc2(12582912.f);  // 1.5 x 2^23
    return (x + m) - m;
}
// The slices of two values, packed FP16.
__device__ __forceinline__ void cut2(f2 x, uint32_t& s1, uint32_t& s2, uint32_t& s3) {
    float a, b;
    const f2 i1 = rint2(x), r1 = x - i1;
    const f2 i2 = rint2(r1 * bc2(kSlice)) * bc2(kUnslice);
    unpk2(i1, a, b);
    s1 = f16x2_rn(a, b);
    unpk2(i2, a, b);
    s2 = f16x2_rn(a, b);
    unpk2(r1 - i2, a, b);
    s3 = f16x2_rn(a, b);
}
__device__ __forceinline__ void cut4(float4 v, float scale, uint2& s1, uint2& s2, uint2& s3) {
    const f2 sc = bc2(scale);
    cut2(mk2(v.x, v.y) * sc, s1.x, s2.x, s3.x);
    cut2(mk2(v.z, v.w) * sc, s1.y, s2.y, s3.y);
}

// ------------------------------------------------------------------ Gram
constexpr int GX_BK = 32, GX_STAGES = 4, GX_SPLIT_WARPS = 16, GX_SPLIT = GX_SPLIT_WARPS * 32;
constexpr int GX_THREADS = GX_SPLIT + 64;
constexpr int GX_F32_TILE = TC_M * GX_BK * 4, GX_F32_STAGE = 2 * GX_F32_TILE;
constexpr int GX_BF_TILE = TC_M * GX_BK * 2, GX_BF_STAGE = 6 * GX_BF_TILE;  // three slices of A, three of B
constexpr int GX_SMEM_BYTES = GX_STAGES * GX_F32_STAGE + 2 * GX_BF_STAGE + 1024;
constexpr int GX_DRAIN = 8;  // steps an accumulation period: 256 points
static_assert(GX_DRAIN * GX_BK <= 256, "a1 b1 <= 2^16: 256 products stay below 2^24");

__device__ __forceinline__ void cut_tile(const unsigned char* f32, unsigned char* dst, float sc0, float sc1) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int e = threadIdx.x + j * GX_SPLIT;
        const int r = e >> 3, kv = (e & 7) * 4;
        const float4 v = *reinterpret_cast<const float4*>(f32 + (size_t)r * (GX_BK * 4) + kv * 4);
        uint2 a, b, c;
        cut4(v, j ? sc1 : sc0, a, b, c);
        const uint32_t off = sw64_off(r, kv);
        *reinterpret_cast<uint2*>(dst + off) = a;
        *reinterpret_cast<uint2*>(dst + GX_BF_TILE + off) = b;
        *reinterpret_cast<uint2*>(dst + 2 * GX_BF_TILE + off) = c;
    }
}

// Add one period's accumulators (32 columns of each order, the two low ones as
// one) into the Kahan sums, the smallest first (compensations as BF16 pairs).
__device__ __forceinline__ void drain_exact(uint32_t taddr, float* fold, uint32_t* comp2) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        uint32_t v[4][8];
#pragma unroll
        for (int o = 0; o < 4; ++o) tmem_ld8(taddr + (3 - o) * TC_N + 8 * h, v[o]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 8; ++j) v[1][j] = __float_as_uint(__uint_as_float(v[1][j]) + __uint_as_float(v[0][j]));
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const int q = 8 * h + j;
            const uint32_t c = comp2[q >> 1];
            float cc[2] = {__uint_as_float(c << 16), __uint_as_float(c & 0xffff0000u)};
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int o = 1; o < 4; ++o) {
                    const float y = __uint_as_float(v[o][j + u]) - cc[u];
                    const float t = fold[q + u] + y;
                    cc[u] = (t - fold[q + u]) - y;
                    fold[q + u] = t;
                }
            comp2[q >> 1] = bf16x2_rn(cc[0], cc[1]);
        }
    }
}

// Warp roles, hand-offs and bounds as in tc_gram_ws_kernel (tc_gemm.cu): warps
// 0-15 cut and drain, warp 16 copies, warp 17 issues the MMAs.
__global__ void __launch_bounds__(GX_THREADS, 1)
    gram_exact_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M, int N,
                      size_t K, size_t kchunk, int tiles_m, bool sym, const unsigned* __restrict__ max_a,
                      const unsigned* __restrict__ max_b, double* __restrict__ work, int* __restrict__ err) {
    extern __shared__ unsigned char tc_smem_raw[];
    __shared__ uint64_t full[GX_STAGES], empty[GX_STAGES], split_bar[2], mma_bar[2], drained_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    __shared__ int last_issued[GX_STAGES];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* f32 = smem;
    unsigned char* bf = smem + GX_STAGES * GX_F32_STAGE;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int tm, tn;
    gram_tile((int)blockIdx.x, tiles_m, sym, tm, tn);
    const bool diag = sym && tm == tn;  // A's slices serve as B's
    const int m0 = tm * TC_M, n0 = tn * TC_N;
    const size_t k_begin = (size_t)blockIdx.z * kchunk;
    const size_t k_end = min(K, k_begin + kchunk);
    const int nsteps = (int)((k_end - k_begin + GX_BK - 1) / GX_BK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < GX_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], GX_SPLIT_WARPS);
            last_issued[s] = -1;
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&split_bar[b], GX_SPLIT_WARPS);
            mbar_init(&mma_bar[b], 1);
        }
        mbar_init(&drained_bar, GX_SPLIT_WARPS);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        // four orders x 128 FP32 columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base_sh)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    int committed = 0;  // MMA thread: steps committed

    if (warp == GX_SPLIT_WARPS) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
            for (int t = 0; t < nsteps; ++t) {
                const int s = t % GX_STAGES;
                if (t >= GX_STAGES && !mbar_wait_or_abort(&empty[s], (uint32_t)(t / GX_STAGES - 1) & 1, &abort_sh)) break;
                const int x = (int)(k_begin + (size_t)t * GX_BK);
                mbar_expect_tx(&full[s], diag ? GX_F32_TILE : GX_F32_STAGE);
                tma_load_2d(f32 + s * GX_F32_STAGE, &map_a, x, m0, &full[s]);
                if (!diag) tma_load_2d(f32 + s * GX_F32_STAGE + GX_F32_TILE, &map_b, x, n0, &full[s]);
                last_issued[s] = t;
            }
        }
    } else if (warp == GX_SPLIT_WARPS + 1) {
        if (lane == 0) {
            for (int t = 0; t < nsteps; ++t) {
                const int b = t & 1;
                if (!mbar_wait_or_abort(&split_bar[b], (uint32_t)(t >> 1) & 1, &abort_sh)) break;
                // a period starts once the last one's sums are read
                if (t > 0 && t % GX_DRAIN == 0 &&
                    !mbar_wait_or_abort(&drained_bar, (uint32_t)(t / GX_DRAIN - 1) & 1, &abort_sh))
                    break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = smem_u32(bf + b * GX_BF_STAGE), bb = diag ? a : a + 3 * GX_BF_TILE;
#pragma unroll
                for (int kk = 0; kk < GX_BK / 16; ++kk)
                    mma_orders<true>(tmem, (t % GX_DRAIN == 0 && kk == 0) ? 0u : 1u,
                                     [&](uint32_t acc, int i, int j, uint32_t first) {
                                         mma_f16(acc, sw64_desc(a + kk * 32 + i * GX_BF_TILE),
                                                 sw64_desc(bb + kk * 32 + j * GX_BF_TILE), first);
                                     });
                mma_commit(&mma_bar[b]);
                committed = t + 1;
            }
        }
    } else {
        float sa[2], sb[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = (threadIdx.x >> 3) + 64 * j;
            sa[j] = m0 + r < M ? pow2f(row_exponent(max_a[m0 + r])) : 1.f;
            sb[j] = n0 + r < N ? pow2f(row_exponent(max_b[n0 + r])) : 1.f;
        }
        float fold[32];
        uint32_t comp2[16];
#pragma unroll
        for (int q = 0; q < 32; ++q) fold[q] = 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) comp2[q] = 0u;
        const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 32);
        bool ok = true;
        for (int t = 0; t < nsteps; ++t) {
            const int s = t % GX_STAGES, b = t & 1;
            if (!mbar_wait_or_abort(&full[s], (uint32_t)(t / GX_STAGES) & 1, &abort_sh)) { ok = false; break; }
            if (t >= 2 && !mbar_wait_or_abort(&mma_bar[b], (uint32_t)((t >> 1) - 1) & 1, &abort_sh)) {
                ok = false;
                break;
            }
            const unsigned char* fs = f32 + s * GX_F32_STAGE;
            unsigned char* bs = bf + b * GX_BF_STAGE;
            cut_tile(fs, bs, sa[0], sa[1]);
            if (!diag) cut_tile(fs + GX_F32_TILE, bs + 3 * GX_BF_TILE, sb[0], sb[1]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&empty[s]);
                mbar_arrive(&split_bar[b]);
            }
            // the period before is complete with the MMAs of step t - 1 (this step's
            // slices are written, so only the MMAs wait for the drain)
            if (t > 0 && t % GX_DRAIN == 0) {
                if (!mbar_wait_or_abort(&mma_bar[b ^ 1], (uint32_t)((t - 1) >> 1) & 1, &abort_sh)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                drain_exact(tlane, fold, comp2);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&drained_bar);
            }
        }
        if (ok && nsteps > 0 &&
            !mbar_wait_or_abort(&mma_bar[(nsteps - 1) & 1], (uint32_t)((nsteps - 1) >> 1) & 1, &abort_sh))
            ok = false;
        if (ok) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (nsteps > 0) drain_exact(tlane, fold, comp2);
            const int row = m0 + (warp & 3) * 32 + lane;
            const int c0 = n0 + (warp >> 2) * 32;
            double* out = work + (size_t)blockIdx.z * M * N + (size_t)row * N;
            if (row < M) {
                const int er = row_exponent(max_a[row]);
#pragma unroll
                for (int q = 0; q < 32; ++q)
                    if (c0 + q < N) {
                        const double v = (double)fold[q] - (double)__uint_as_float((q & 1) ? (comp2[q >> 1] & 0xffff0000u)
                                                                                           : (comp2[q >> 1] << 16));
                        const int e = er + row_exponent(max_b[c0 + q]);
                        out[c0 + q] = v * __longlong_as_double((long long)(1023 - e) << 52);
                    }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_sh) {
        // drain: copies still landing, MMAs still running (bounded waits)
        if (warp == GX_SPLIT_WARPS && lane == 0)
            for (int s = 0; s < GX_STAGES; ++s)
                if (last_issued[s] >= 0) mbar_wait(&full[s], (uint32_t)(last_issued[s] / GX_STAGES) & 1);
        if (warp == GX_SPLIT_WARPS + 1 && lane == 0 && committed > 0)
            mbar_wait(&mma_bar[(committed - 1) & 1], (uint32_t)((committed - 1) >> 1) & 1);
        if (threadIdx.x == 0) atomicExch(err, 1);
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ------------------------------------------------------------------ rotation
constexpr int CX_N = TC_N;

// Slices of the coefficients, [slice][npad][kpad] FP16 (targets by rows, zero
// padded): column n of coef[k][n] 2^-e_k (the rows of A are scaled by 2^e_k),
// brought to below 256 by a power of two.  scale_a[k]: 2^e_k (padding: 0),
// scale_out[n]: the inverse of column n's power.
__global__ void coef_cut_kernel(int Kc, int N, const double* __restrict__ coef, int ldcoef, int kpad, int npad,
                                const unsigned* __restrict__ max_a, __half* __restrict__ out, float* __restrict__ scale_a,
                                float* __restrict__ scale_out) {
    __shared__ double sh[32];
    const int n = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto value = [&](int k) {
        return n < N && k < Kc ? ldexp(coef[(size_t)k * ldcoef + n], -row_exponent(max_a[k])) : 0.0;
    };
    double m = 0.0;
    for (int k = threadIdx.x; k < Kc; k += blockDim.x) m = fmax(m, fabs(value(k)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) sh[warp] = m;
    __syncthreads();
    m = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, sh[w]);
    int e = 0;
    if (m > 0.0 && m < INFINITY) {
        frexp(m, &e);  // m < 2^e
        e = 8 - e;
    }
    e = e < -126 ? -126 : e > 126 ? 126 : e;
    if (threadIdx.x == 0) scale_out[n] = pow2f(-e);
    if (n == 0)
        for (int k = threadIdx.x; k < kpad; k += blockDim.x) scale_a[k] = k < Kc ? pow2f(row_exponent(max_a[k])) : 0.f;
    for (int k = threadIdx.x; k < kpad; k += blockDim.x) {
        const double x = ldexp(value(k), e);
        const double i1 = rint(x), r1 = x - i1, i2 = rint(r1 * 512.0) / 512.0;
        const size_t at = (size_t)n * kpad + k, step = (size_t)npad * kpad;
        out[at] = __float2half_rn((float)i1);
        out[at + step] = __float2half_rn((float)i2);
        out[at + 2 * step] = __double2half(r1 - i2);
    }
}

// Three FP16 slices, their eight products by order in three accumulators.
struct ExactSlices {
    static constexpr int SLICES = 3, ACCS = 3;
    static constexpr bool SCALED = true;
    static constexpr uint32_t FORMAT = 0;  // F16
    static __device__ __forceinline__ void cut(f2 x, uint32_t* s) { cut2(x, s[0], s[1], s[2]); }
    template <class Mma> static __device__ __forceinline__ void products(uint32_t acc, uint32_t first, Mma mma) {
        mma_orders<false>(acc, first, mma);
    }
};

// ------------------------------------------------------------------ row maxima
// out[row] = bits of the largest finite |x| of the row (zeroed before; infinities
// and NaN reach the results at their own points whatever the scale, and must not set
// that of the other points); Tin = double: the row is also rounded to FP32 into
// dst (the load's conversion).
template <typename Tin>
__global__ void row_max_kernel(const Tin* __restrict__ src, float* __restrict__ dst, size_t n, unsigned* __restrict__ out) {
    const size_t row = blockIdx.y, q4 = n / 4;
    const Tin* s = src + row * n;
    float* d = dst + row * n;
    float m = 0.f;
    auto use = [&](float x) { m = fabsf(x) < INFINITY ? fmaxf(m, fabsf(x)) : m; };
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < q4; q += (size_t)gridDim.x * blockDim.x) {
        float4 v;
        if constexpr (sizeof(Tin) == 8) {
            const double2 a = __ldg(reinterpret_cast<const double2*>(s) + 2 * q), b = __ldg(reinterpret_cast<const double2*>(s) + 2 * q + 1);
            v = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
            reinterpret_cast<float4*>(d)[q] = v;
        } else {
            v = __ldg(reinterpret_cast<const float4*>(s) + q);
        }
        use(v.x);
        use(v.y);
        use(v.z);
        use(v.w);
    }
    const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0 && w) atomicMax(out + row, w);
}

size_t exact_tiles(int M, int N, bool sym) {
    const size_t tm = (M + TC_M - 1) / TC_M, tn = (N + TC_N - 1) / TC_N;
    return sym ? tm * (tm + 1) / 2 : tm * tn;
}
// K chunks: one wave of CTAs (one an SM), at least 256 points each.
size_t exact_chunks(int M, int N, size_t K, bool sym) {
    const size_t want = std::max<size_t>(1, 152 / exact_tiles(M, N, sym));
    return std::max<size_t>(1, std::min(want, (K + 255) / 256));
}

}  // namespace

bool exact_ok(size_t K, const void* a) { return K % 4 == 0 && K <= 0x7fffffffull && (uintptr_t)a % 16 == 0 && encode_tiled() != nullptr; }

cudaError_t convert_row_max(const double* in, float* out, int rows, size_t n, unsigned* d_max, cudaStream_t s, int* launches) {
    cudaError_t e = cudaMemsetAsync(d_max, 0, sizeof(unsigned) * rows, s);
    if (e || rows == 0) return e;
    const unsigned per = (unsigned)std::max<size_t>(1, std::min<size_t>((n / 4 + 511) / 512, (152 * 16 + rows - 1) / rows));
    row_max_kernel<double><<<dim3(per, rows), 256, 0, s>>>(in, out, n, d_max);
    *launches += 1;
    return cudaGetLastError();
}
cudaError_t row_max(const float* in, int rows, size_t n, unsigned* d_max, cudaStream_t s, int* launches) {
    cudaError_t e = cudaMemsetAsync(d_max, 0, sizeof(unsigned) * rows, s);
    if (e || rows == 0) return e;
    const unsigned per = (unsigned)std::max<size_t>(1, std::min<size_t>((n / 4 + 511) / 512, (152 * 16 + rows - 1) / rows));
    row_max_kernel<float><<<dim3(per, rows), 256, 0, s>>>(in, nullptr, n, d_max);
    *launches += 1;
    return cudaGetLastError();
}

size_t gram_exact_work_elems(int M, int N, size_t K, bool sym) { return exact_chunks(M, N, K, sym) * (size_t)M * N; }

cudaError_t gram_exact(int M, int N, size_t K, const float* A, const unsigned* max_a, const float* B, const unsigned* max_b,
                       double alpha, double* C, int ldc, double* work, size_t work_elems, int* d_err, cudaStream_t s,
                       int* launches) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    const bool sym = A == B && M == N;
    const size_t nch = exact_chunks(M, N, K, sym);
    if (!exact_ok(K, A) || !exact_ok(K, B) || nch * (size_t)M * N > work_elems) return cudaErrorInvalidValue;
    size_t kchunk = (K + nch - 1) / nch;
    kchunk = (kchunk + GX_BK - 1) / GX_BK * GX_BK;
    const size_t nch_eff = (K + kchunk - 1) / kchunk;
    CUtensorMap map_a, map_b;
    auto map = [&](CUtensorMap* m, const float* p, int rows) {
        return make_map(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sizeof(float), p, (size_t)rows, K, K, GX_BK, TC_M,
                        CU_TENSOR_MAP_SWIZZLE_NONE);
    };
    if (!map(&map_a, A, M) || !map(&map_b, B, N)) return cudaErrorInvalidValue;
    static std::atomic<unsigned long long> attr_done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    cudaError_t e;
    if (dev >= 64 || !(attr_done.load() & (1ull << dev))) {
        if ((e = cudaFuncSetAttribute(gram_exact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GX_SMEM_BYTES))) return e;
        if (dev < 64) attr_done.fetch_or(1ull << dev);
    }
    if ((e = cudaMemsetAsync(d_err, 0, sizeof(int), s))) return e;
    gram_exact_kernel<<<dim3((unsigned)exact_tiles(M, N, sym), 1, (unsigned)nch_eff), GX_THREADS, GX_SMEM_BYTES, s>>>(
        map_a, map_b, M, N, K, kchunk, (M + TC_M - 1) / TC_M, sym, max_a, max_b, work, d_err);
    *launches += 2;
    return chunk_sum(M, N, nch_eff, work, alpha, sym, TC_M, C, ldc, s);
}

size_t combine_exact_scratch_bytes(int N, int Kc) {
    const size_t kpad = ((size_t)Kc + CW_BK - 1) / CW_BK * CW_BK, npad = ((size_t)N + CX_N - 1) / CX_N * CX_N;
    return 3 * kpad * npad * sizeof(__half) + (npad + kpad) * sizeof(float);
}

cudaError_t combine_exact(int N, size_t K, int Kc, const float* A, const unsigned* max_a, const double* Coef, int ldcoef,
                          bool add, float* Out, size_t ldo, void* scratch, int* d_err, cudaStream_t s, int* launches) {
    if (N <= 0 || K == 0) return cudaSuccess;
    if (!exact_ok(K, A) || Kc <= 0) return cudaErrorInvalidValue;
    const int kpad = (Kc + CW_BK - 1) / CW_BK * CW_BK, npad = (N + CX_N - 1) / CX_N * CX_N;
    __half* slices = static_cast<__half*>(scratch);
    float* scale_a = reinterpret_cast<float*>(slices + (size_t)3 * kpad * npad);
    float* scale_out = scale_a + kpad;
    CUtensorMap map_a, map_c;
    if (!make_map(&map_a, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sizeof(float), A, (size_t)Kc, K, K, TC_M, CW_BK,
                  CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map(&map_c, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, slices, (size_t)3 * npad, (size_t)kpad, (size_t)kpad, CW_BK, CX_N,
                  CU_TENSOR_MAP_SWIZZLE_64B))
        return cudaErrorInvalidValue;
    static std::atomic<unsigned long long> attr_done{0};
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e;
    if (dev >= 64 || !(attr_done.load() & (1ull << dev))) {
        if ((e = cudaFuncSetAttribute(combine_ws_kernel<ExactSlices, CX_N, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, CombineShape<ExactSlices, CX_N>::SMEM))) return e;
        if (dev < 64) attr_done.fetch_or(1ull << dev);
    }
    if ((e = cudaMemsetAsync(d_err, 0, sizeof(int), s))) return e;
    coef_cut_kernel<<<npad, 128, 0, s>>>(Kc, N, Coef, ldcoef, kpad, npad, max_a, slices, scale_a, scale_out);
    bool resident;
    const unsigned grid = combine_grid<ExactSlices, CX_N>(N, K, kpad, npad, sms, &resident);
    combine_ws_kernel<ExactSlices, CX_N, float><<<grid, CW_THREADS, CombineShape<ExactSlices, CX_N>::SMEM, s>>>(
        map_a, map_c, N, K, kpad, npad, scale_a, scale_out, resident, add ? 1.f : 0.f, Out, ldo, d_err);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace lace
