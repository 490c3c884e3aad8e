// Combinations over orbitals Out[n][r] = beta Out[n][r] + sum_k Coef[k][n] A[k][r]
// on the tensor cores, for the slice schemes of tc_exact.cu and tc_gemm.cu: tiles of
// 128 points x NT targets, 32 orbitals a step, persistent over tiles.  The FP32
// rows [k][r] and the cut coefficients [slice][n][k] come by TMA; the rows' slices go to
// TMEM, a point a lane, so that shared memory feeds the MMAs with one operand only.
// A step's coefficients are as many bytes as its rows or more, so they stay in shared
// memory for all tiles of a CTA where they fit.
//
// Measured, 72^3 x 256 -> 256 in two BF16 slices (launches, alone): FP32 output 200
// -> 188 us, FP64 308 -> 281 (147 and 220 us at the rate of a plain copy of these
// rows); to 64 targets in FP64 179 -> 145 us (110): against a CTA-wide barrier a step
// and A's slices in shared memory.  Three FP16 slices (eight products): 420 -> 225 us.
// What is left is each step's chain of hand-offs, and the cut waiting while a tile's
// results are stored.
#pragma once

#include <algorithm>
#include <numeric>

#include "f32x2.cuh"
#include "tc_util.cuh"

namespace lace {
namespace {

constexpr int CW_BK = 32, CW_CUT_WARPS = 16, CW_AHEAD = 2;
constexpr int CW_THREADS = CW_CUT_WARPS * 32 + 64;
constexpr int CW_A32_BYTES = CW_BK * TC_M * 4;  // 16 KB: 32 orbitals x 128 points
constexpr int CW_A_COLS = CW_BK / 2;            // TMEM columns of a slice of A

// Slice scheme S: SLICES (FORMAT: the MMA's operand type), the accumulators ACCS, the
// products, SCALED (powers of two on rows and targets).
template <class S, int NT> struct CombineShape {
    static constexpr int B_TILE = NT * CW_BK * 2, B_BYTES = S::SLICES * B_TILE;
    // Stages of rows: an even number, so that a stage passes between steps of one set of
    // cut warps (below).  With five, a set could wait for a stage whose rows of the other
    // set's step had not landed: a wait knows only the parity of a phase, took the phase
    // before last for the awaited one, and the stage was read with other rows and freed early
    // (rows landing out of order by two steps, so under load from other streams).  Six are as
    // fast as five were, four up to 4% slower (80^3 x 512 -> 128: 454, 462, 488 us).
    static constexpr int ASTAGES = 6;
    static constexpr int BSTAGES = (227 * 1024 - 1536 - ASTAGES * CW_A32_BYTES) / B_BYTES;
    static constexpr int SMEM = BSTAGES * B_BYTES + ASTAGES * CW_A32_BYTES + 1024;
    // TMEM columns: the accumulators, then up to four stages of A's slices
    static constexpr int A_AT = S::ACCS * NT, A_STAGE = S::SLICES * CW_A_COLS;
    static constexpr int TSTAGES = (512 - A_AT) / A_STAGE < 4 ? 2 : 4;
    static constexpr int COLS = A_AT + TSTAGES * A_STAGE <= 256 ? 256 : 512;
    static constexpr uint32_t IDESC =
        (1u << 4) | (S::FORMAT << 7) | (S::FORMAT << 10) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
    static_assert(SMEM <= 227 * 1024 - 512, "one CTA an SM");
    static_assert(TSTAGES >= 2 && TSTAGES % 2 == 0 && CW_BK == 16 * (CW_CUT_WARPS / 8), "slice stages; 16 orbitals a thread");
    static_assert(ASTAGES > CW_AHEAD && ASTAGES % 2 == 0, "rows ahead; the steps of a set alone in a stage");
};

// D (FP32) += A B^T with A in TMEM (a point a lane, two orbitals a 32-bit column).
template <uint32_t IDESC>
__device__ __forceinline__ void mma_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(IDESC), "r"(accumulate));
}
// 8 FP32 accumulator columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// Warp roles: warps 0-15 cut the FP32 rows into A's slices in TMEM and write the
// results, warp 16 copies, warp 17 issues the MMAs.  Warps 0-7 cut the even steps
// and 8-15 the odd ones (warp w: points 32 (w % 4).., orbitals 16 (w / 4 % 2).. of
// a step), so that two steps' chains of load, cut, store and wait overlap.  Hand-offs by
// mbarriers: full_a/full_b (copies landed), empty_a (a stage of rows is cut), cut_bar
// (slices are in TMEM), mma_bar (the MMAs are done with a slice stage), empty_b (and
// with their coefficients), tile_bar (and with a tile), drained_bar (a tile's sums are in registers; its stores
// run under the next tile's MMAs).
template <class S, int NT, typename TO>
__global__ void __launch_bounds__(CW_THREADS, 1)
    combine_ws_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_c, int N, size_t K,
                      int kpad, int npad, const float* __restrict__ scale_a, const float* __restrict__ scale_out,
                         bool resident, float beta,
                      TO* __restrict__ Out, size_t ldo, int* __restrict__ err) {
    using C = CombineShape<S, NT>;
    extern __shared__ unsigned char tc_smem_raw[];
    __shared__ uint64_t full_a[C::ASTAGES], empty_a[C::ASTAGES], full_b[C::BSTAGES], empty_b[C::BSTAGES];
    __shared__ uint64_t cut_bar[C::TSTAGES], mma_bar[C::TSTAGES], tile_bar, drained_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    __shared__ int last_a[C::ASTAGES], last_b[C::BSTAGES];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* bst = smem;                           // coefficient slices
    unsigned char* a32 = bst + C::BSTAGES * C::B_BYTES;  // FP32 rows
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nsteps = kpad / CW_BK;
    const int rtiles = (int)((K + TC_M - 1) / TC_M), ntiles = npad / NT;
    const long long tiles = (long long)rtiles * ntiles;
    const int my_tiles = (int)((tiles - 1 - (long long)blockIdx.x) / (int)gridDim.x + 1);  // gridDim.x <= tiles
    const int total = my_tiles * nsteps;  // this CTA's steps over all its tiles
    // step g is orbital step g % nsteps of tile g / nsteps of this CTA (targets
    // fastest: the tiles of the same points run side by side).  resident: all steps'
    // coefficients fit the stages and this CTA's tiles have the same targets (the
    // grid is a multiple of ntiles), so they are copied once.
    auto tile_of_step = [&](int g, int& rt, int& nt) {
        const long long tile = (long long)blockIdx.x + (long long)(g / nsteps) * (int)gridDim.x;
        rt = (int)(tile / ntiles);
        nt = (int)(tile % ntiles);
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::ASTAGES; ++s) {
            mbar_init(&full_a[s], 1);
            mbar_init(&empty_a[s], CW_CUT_WARPS / 2);
            last_a[s] = -1;
        }
        for (int s = 0; s < C::BSTAGES; ++s) {
            mbar_init(&full_b[s], 1);
            mbar_init(&empty_b[s], 1);
            last_b[s] = -1;
        }
        for (int s = 0; s < C::TSTAGES; ++s) {
            mbar_init(&cut_bar[s], CW_CUT_WARPS / 2);
            mbar_init(&mma_bar[s], 1);
        }
        mbar_init(&tile_bar, 1);
        mbar_init(&drained_bar, CW_CUT_WARPS);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base_sh)),
                     "r"(C::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    int committed = 0;  // MMA thread: steps committed

    if (warp == CW_CUT_WARPS) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_c)) : "memory");
            // the rows run CW_AHEAD steps ahead of the coefficients (HBM and L2)
            for (int g = -CW_AHEAD; g < total; ++g) {
                int rt, nt;
                const int ga = g + CW_AHEAD;
                if (ga < total) {
                    const int sa = ga % C::ASTAGES;
                    tile_of_step(ga, rt, nt);
                    if (ga >= C::ASTAGES && !mbar_wait_or_abort(&empty_a[sa], (uint32_t)(ga / C::ASTAGES - 1) & 1, &abort_sh)) break;
                    mbar_expect_tx(&full_a[sa], CW_A32_BYTES);
                    tma_load_2d(a32 + sa * CW_A32_BYTES, &map_a, rt * TC_M, (ga % nsteps) * CW_BK, &full_a[sa]);
                    last_a[sa] = ga;
                }
                if (g < 0 || (resident && g >= nsteps)) continue;
                const int sb = g % C::BSTAGES;
                tile_of_step(g, rt, nt);
                if (g >= C::BSTAGES && !mbar_wait_or_abort(&empty_b[sb], (uint32_t)(g / C::BSTAGES - 1) & 1, &abort_sh)) break;
                mbar_expect_tx(&full_b[sb], C::B_BYTES);
#pragma unroll
                for (int q = 0; q < S::SLICES; ++q)
                    tma_load_2d(bst + sb * C::B_BYTES + q * C::B_TILE, &map_c, (g % nsteps) * CW_BK, q * npad + nt * NT,
                                &full_b[sb]);
                last_b[sb] = g;
            }
        }
    } else if (warp == CW_CUT_WARPS + 1) {
        if (lane == 0) {
            for (int g = 0; g < total; ++g) {
                const int b = g % C::TSTAGES, step = g % nsteps, sb = resident ? step : g % C::BSTAGES;
                if (!mbar_wait_or_abort(&full_b[sb], resident ? 0u : (uint32_t)(g / C::BSTAGES) & 1, &abort_sh) ||
                    !mbar_wait_or_abort(&cut_bar[b], (uint32_t)(g / C::TSTAGES) & 1, &abort_sh))
                    break;
                // a tile starts once the last one's sums are read
                if (g > 0 && step == 0 && !mbar_wait_or_abort(&drained_bar, (uint32_t)(g / nsteps - 1) & 1, &abort_sh)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = tmem + C::A_AT + b * C::A_STAGE, bb = smem_u32(bst + sb * C::B_BYTES);
#pragma unroll
                for (int kk = 0; kk < CW_BK / 16; ++kk)
                    S::products(tmem, (step == 0 && kk == 0) ? 0u : 1u, [&](uint32_t acc, int i, int j, uint32_t first) {
                        mma_ta<C::IDESC>(acc, a + i * CW_A_COLS + kk * 8, sw64_desc(bb + kk * 32 + j * C::B_TILE), first);
                    });
                mma_commit(&mma_bar[b]);
                if (!resident) mma_commit(&empty_b[sb]);
                if (step == nsteps - 1) mma_commit(&tile_bar);
                committed = g + 1;
            }
            // The commits of a step may arrive in any order: none may be on its way when
            // the CTA leaves (the others are waited for by the next users of their stages).
            for (int g = max(0, committed - C::TSTAGES); g < committed; ++g)
                mbar_wait(&mma_bar[g % C::TSTAGES], (uint32_t)(g / C::TSTAGES) & 1);
            for (int g = max(0, committed - C::BSTAGES); g < committed && !resident; ++g)
                mbar_wait(&empty_b[g % C::BSTAGES], (uint32_t)(g / C::BSTAGES) & 1);
        }
    } else {
        const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int ar = (warp & 3) * 32 + lane, set = warp >> 3, kq = (warp >> 2 & 1) * 16, cb = (warp >> 2) * (NT / 4);
        // the sums of the tile that ends with step g -> Out (NT / 4 targets of one point a thread)
        auto finish_tile = [&](int g, bool more) {
            if (!mbar_wait_or_abort(&tile_bar, (uint32_t)(g / nsteps) & 1, &abort_sh)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float x[NT / 4];
#pragma unroll
            for (int h = 0; h < NT / 32; ++h) {
                uint32_t v[S::ACCS][8];
#pragma unroll
                for (int o = 0; o < S::ACCS; ++o) tmem_ld8(tlane + o * NT + cb + 8 * h, v[o]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float t = __uint_as_float(v[S::ACCS - 1][j]);
#pragma unroll
                    for (int o = S::ACCS - 2; o >= 0; --o) t = __uint_as_float(v[o][j]) + t;
                    x[8 * h + j] = t;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (more && lane == 0) mbar_arrive(&drained_bar);
            int rt, nt;
            tile_of_step(g, rt, nt);
            const size_t r = (size_t)rt * TC_M + ar;
            const int n0 = nt * NT + cb;
            if (r < K) {
#pragma unroll
                for (int j = 0; j < NT / 4; ++j)
                    if (n0 + j < N) {
                        TO* o = Out + (size_t)(n0 + j) * ldo + r;
                        const float y = S::SCALED ? x[j] * __ldg(scale_out + n0 + j) : x[j];
                        *o = beta == 0.f ? (TO)y : (TO)(beta * (float)*o + y);
                    }
            }
            return true;
        };
        auto cut_step = [&](int g) {
            const int sa = g % C::ASTAGES, b = g % C::TSTAGES, k0 = g % nsteps * CW_BK + kq;
            float4 c[4];
            if (S::SCALED)
#pragma unroll
                for (int i = 0; i < 4; ++i) c[i] = __ldg(reinterpret_cast<const float4*>(scale_a + k0) + i);
            if (!mbar_wait_or_abort(&full_a[sa], (uint32_t)(g / C::ASTAGES) & 1, &abort_sh)) return false;
            // the MMAs of step g - TSTAGES are done with slice stage b
            if (g >= C::TSTAGES && !mbar_wait_or_abort(&mma_bar[b], (uint32_t)(g / C::TSTAGES - 1) & 1, &abort_sh)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const float* src = reinterpret_cast<const float*>(a32 + sa * CW_A32_BYTES) + kq * TC_M + ar;
            uint32_t s[S::SLICES][8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                f2 x = mk2(src[(2 * q) * TC_M], src[(2 * q + 1) * TC_M]);
                if (S::SCALED) x = x * (q & 1 ? mk2(c[q >> 1].z, c[q >> 1].w) : mk2(c[q >> 1].x, c[q >> 1].y));
                uint32_t t[S::SLICES];
                S::cut(x, t);
#pragma unroll
                for (int i = 0; i < S::SLICES; ++i) s[i][q] = t[i];
            }
            const uint32_t ta = tlane + C::A_AT + b * C::A_STAGE + kq / 2;
#pragma unroll
            for (int i = 0; i < S::SLICES; ++i) tmem_st8(ta + i * CW_A_COLS, s[i]);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&empty_a[sa]);
                mbar_arrive(&cut_bar[b]);
            }
            return true;
        };
        bool ok = true;
        for (int t = 0; t < my_tiles && ok; ++t) {
            bool last = t == 0;  // the tile before is written
            for (int g = t * nsteps + ((t * nsteps ^ set) & 1); g < (t + 1) * nsteps && ok; g += 2) {
                ok = cut_step(g);
                // the tile before, once this step's slices are written (only MMAs wait)
                if (ok && !last) ok = finish_tile(t * nsteps - 1, true), last = true;
            }
            if (ok && !last) ok = finish_tile(t * nsteps - 1, true);
        }
        if (ok) finish_tile(total - 1, false);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_sh) {
        // copies still landing (bounded waits; the MMAs are done)
        if (warp == CW_CUT_WARPS && lane == 0) {
            for (int s = 0; s < C::ASTAGES; ++s)
                if (last_a[s] >= 0) mbar_wait(&full_a[s], (uint32_t)(last_a[s] / C::ASTAGES) & 1);
            for (int s = 0; s < C::BSTAGES; ++s)
                if (last_b[s] >= 0) mbar_wait(&full_b[s], (uint32_t)(last_b[s] / C::BSTAGES) & 1);
        }
        if (threadIdx.x == 0) atomicExch(err, 1);
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::COLS) : "memory");
    }
}

// The grid of a combination: one CTA an SM, the coefficients resident where they
// fit.  Where they do not and the last tile of targets is mostly padding, the grid shares
// no factor with their number, so that every CTA takes its part of the short tiles
// (72^3 x 320 -> 320 in FP64 612 -> 525 us: half of the CTAs had full tiles alone).
template <class S, int NT> unsigned combine_grid(int N, size_t K, int kpad, int npad, int sms, bool* resident) {
    const long long ntiles = npad / NT, tiles = (long long)((K + TC_M - 1) / TC_M) * ntiles;
    *resident = kpad / CW_BK <= CombineShape<S, NT>::BSTAGES && ntiles <= sms;
    if (*resident) return (unsigned)std::min<long long>(tiles, sms / ntiles * ntiles);
    long long grid = std::min<long long>(tiles, sms);
    while (npad - N >= NT / 4 && grid > 1 && std::gcd(grid, ntiles) > 1) --grid;
    return (unsigned)grid;
}

}  // namespace
}  // namespace lace
