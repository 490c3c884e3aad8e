// Pivoted QR of the SCDM subsample (Sec. 2) in rounds: one persistent
// cooperative launch whose CTAs meet a few times a round instead of once a
// pivot.
//
// The norms of the residual columns only fall, so what a column's norm was at
// the start of a round bounds it until the end.  A round brings all norms up
// to date with the directions of the last round, takes the columns with the
// largest norms as candidates (at most kCand, all above a bound tau that no
// other column reaches), and one CTA then selects pivots among the candidates
// alone for as long as their largest residual norm stays above tau: each is
// the column that the step-by-step algorithm would pick (largest norm, ties
// to the lowest index).  In localised systems a pivot takes only its
// neighbourhood down: at 72^3 with 256 orbitals a round yields its 64 pivots.
//
// A round:
//   A  norms: n_j -= sum (q . v_j)^2 over the directions of the last round, an
//      FP32 product of the new directions with all columns on packed pairs
//      (the columns themselves are never rewritten; norms are kept in FP64)
//   B  histogram of the norms within a factor of 4 of the largest
//   C  tau and the list of candidates
//   D  the candidates' residuals v - Q Q^T v
//   E  their Gram matrix
//   F  CTA 0: pivoted Cholesky of the Gram matrix (the candidates' residual
//      norms on its diagonal) until tau, then the new directions from the
//      pivots' residuals and the factor
// The matrix is read from L2 or HBM once a round where the step-by-step
// kernels went through (and, off chip, rewrote) it once a pivot.
#pragma once

#include "f32x2.cuh"
#include "grid_sync.cuh"
#include "lace_internal.cuh"

namespace lace {
namespace qrr {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kCand = 512;      // candidates a round, one a thread of CTA 0
constexpr int kSteps = 64;      // pivots a round
constexpr int kBins = 1024;     // histogram: 512 bins an octave of squared norm, two octaves
constexpr int kMaxRows = 1024;
// phase A: a CTA takes 128 columns at a time; each of its four teams of 128
// threads a quarter of the rows, 16 rows a stage, 8 directions x 8 columns a
// thread
constexpr int kTile = 128, kTeams = 4, kChunk = 16, kStages = 3;
constexpr int kStageFloats = kChunk * (kTile + kSteps);
constexpr int kLPitch = kSteps + 4;  // floats a candidate's factor row

struct Buf {
    double* nrm;     // [ncol] squared residual norms; chosen: -1
    float* Q;        // [npiv][nrowp] directions
    float* QT;       // [nrowp][kSteps] the last round's, by row
    int* cand;       // [kCand] column of each candidate
    float* R;        // [kCand][nrowp] candidates' residuals
    float* G;        // [kCand][kCand] Gram matrix
    unsigned* hist;  // [kBins]
    unsigned* ctl;   // [16]
};
// ctl words, by round parity: 0/1 largest norm (float bits), 2/3 candidate
// count, 4/5 lowest index of a single-candidate round; 6 pivots so far

__host__ __device__ inline int padded_rows(int nrow) { return (nrow + 31) / 32 * 32; }

inline size_t align_up(size_t b) { return (b + 255) / 256 * 256; }
template <class F> inline void layout(int nrow, int ncol, F take) {
    const size_t np = padded_rows(nrow);
    take(sizeof(double) * (size_t)ncol);
    take(4 * np * nrow);
    take(4 * np * kSteps);
    take(4 * (size_t)kCand);
    take(4 * np * kCand);
    take(4 * (size_t)kCand * kCand);
    take(4 * (size_t)kBins);
    take(64);
}
inline size_t buf_bytes(int nrow, int ncol) {
    size_t b = 0;
    layout(nrow, ncol, [&](size_t n) { b += align_up(n); });
    return b;
}
inline Buf buf_at(void* p, int nrow, int ncol) {
    void* at[8];
    int i = 0;
    unsigned char* b = static_cast<unsigned char*>(p);
    layout(nrow, ncol, [&](size_t n) {
        at[i++] = b;
        b += align_up(n);
    });
    return Buf{(double*)at[0], (float*)at[1], (float*)at[2], (int*)at[3], (float*)at[4], (float*)at[5], (unsigned*)at[6], (unsigned*)at[7]};
}

// Dynamic shared memory: phase A (the teams' stages, then their partial
// dots), D (partial residuals of every warp), E (two blocks of 32 candidates,
// 256 rows at a time) or F (factor rows of the candidates, the last eight
// steps' entries, the pivots' part of the factor).
__host__ __device__ inline size_t smem_bytes() {
    const size_t a = 4 * (size_t)kTeams * kStages * kStageFloats, p = 4 * (size_t)kTeams * kSteps * kTile;
    const size_t d = 4 * (size_t)kWarps * kMaxRows, e = 4 * 64 * (size_t)(256 + 4);
    const size_t f = 4 * ((size_t)kCand * kLPitch + 8 * kCand + kSteps * kSteps);
    size_t m = a;
    for (size_t x : {p, d, e, f}) m = x > m ? x : m;
    return m;
}

__device__ __forceinline__ unsigned fbits(double n) { return __float_as_uint((float)n); }
__device__ __forceinline__ double ld_nrm(const double* p) { return __ldcg(p); }
__device__ __forceinline__ void team_bar(int team) { asm volatile("bar.sync %0, 128;" ::"r"(1 + team) : "memory"); }
__device__ __forceinline__ void copy16(unsigned dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy4(unsigned dst, const void* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Phase A for the columns c0 .. c0 + 127: returns, to threads 0 .. 127, the
// drop of column c0 + tid: sum over the last round's directions of (q . v)^2.
__device__ __forceinline__ float norm_drop(const float* __restrict__ V, int nrow, int ncol, const Buf& B, int c0, bool vec,
                                           float* smem, float* red) {
    const int tid = threadIdx.x, team = tid >> 7, tt = tid & 127;
    const int quarter = ((nrow + kTeams - 1) / kTeams + kChunk - 1) / kChunk * kChunk;
    const int r0 = team * quarter, r1 = min(nrow, r0 + quarter);
    const int chunks = r1 > r0 ? (r1 - r0 + kChunk - 1) / kChunk : 0;
    float* stage = smem + team * kStages * kStageFloats;
    const unsigned stage_s = (unsigned)__cvta_generic_to_shared(stage);
    auto issue = [&](int t) {
        if (t < chunks) {
            const unsigned st = stage_s + 4u * (t % kStages) * kStageFloats;
            const int r = r0 + t * kChunk;
            if (vec) {
#pragma unroll
                for (int u = 0; u < kChunk * kTile / 4 / 128; ++u) {
                    const int e = tt + u * 128, row = e / (kTile / 4), q = e % (kTile / 4);
                    const bool in = r + row < r1 && c0 + 4 * q < ncol;
                    copy16(st + 16u * e, in ? V + (size_t)(r + row) * ncol + c0 + 4 * q : V, in ? 16 : 0);
                }
            } else {
#pragma unroll 4
                for (int u = 0; u < kChunk * kTile / 128; ++u) {
                    const int row = u, c = c0 + tt;
                    const bool in = r + row < r1 && c < ncol;
                    copy4(st + 4u * (row * kTile + tt), in ? V + (size_t)(r + row) * ncol + c : V, in ? 4 : 0);
                }
            }
#pragma unroll
            for (int u = 0; u < kChunk * kSteps / 4 / 128; ++u) {
                const int e = tt + u * 128;  // (rows past nrow: zeros)
                copy16(st + 4u * kChunk * kTile + 16u * e, B.QT + (size_t)r * kSteps + 4 * e, 16);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int cg = tt & 15, qg = tt >> 4;  // columns 4 cg .. + 3 and 64 + 4 cg .. + 3, directions 8 qg .. + 7
    f2 acc[8][4];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[q][c] = bc2(0.f);
    issue(0);
    issue(1);
    for (int t = 0; t < chunks; ++t) {
        issue(t + 2);
        asm volatile("cp.async.wait_group 2;" ::: "memory");
        team_bar(team);
        const float* vs = stage + (t % kStages) * kStageFloats;
        const float* qs = vs + kChunk * kTile;
#pragma unroll
        for (int r = 0; r < kChunk; ++r) {
            const ulonglong2 va = *reinterpret_cast<const ulonglong2*>(vs + r * kTile + 4 * cg);
            const ulonglong2 vb = *reinterpret_cast<const ulonglong2*>(vs + r * kTile + 64 + 4 * cg);
            const float4 qa = *reinterpret_cast<const float4*>(qs + r * kSteps + 8 * qg);
            const float4 qb = *reinterpret_cast<const float4*>(qs + r * kSteps + 8 * qg + 4);
            const float q[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const f2 w = bc2(q[i]);
                acc[i][0] = fma2(w, f2{va.x}, acc[i][0]);
                acc[i][1] = fma2(w, f2{va.y}, acc[i][1]);
                acc[i][2] = fma2(w, f2{vb.x}, acc[i][2]);
                acc[i][3] = fma2(w, f2{vb.y}, acc[i][3]);
            }
        }
        team_bar(team);  // the stage is refilled by issue(t + 3)
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float* part = smem + (size_t)team * kSteps * kTile;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        ulonglong2* o = reinterpret_cast<ulonglong2*>(part + (8 * qg + i) * kTile);
        o[cg] = make_ulonglong2(acc[i][0].v, acc[i][1].v);
        o[16 + cg] = make_ulonglong2(acc[i][2].v, acc[i][3].v);
    }
    __syncthreads();
    {
        // thread (team, tt): column tt, directions 16 team .. + 15
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < kSteps / kTeams; ++i) {
            const float* o = smem + (team * (kSteps / kTeams) + i) * kTile + tt;
            const float d = (o[0] + o[kSteps * kTile]) + (o[2 * kSteps * kTile] + o[3 * kSteps * kTile]);
            s = fmaf(d, d, s);
        }
        red[tid] = s;
    }
    __syncthreads();
    return tid < kTile ? (red[tid] + red[tid + 128]) + (red[tid + 256] + red[tid + 384]) : 0.f;
}

// Forward substitution of one row from step I on: q_I final, then its share
// taken from the later ones (Lt[I][l] = L[pivot l][step I], zero for l <= I).
template <int I>
__device__ __forceinline__ void solve_step(float (&q)[kSteps], int s, const float* Lt, const float* inv, float* Q, int nrowp) {
    if (I < s) {
        q[I] *= inv[I];
#pragma unroll
        for (int b = (I + 1) / 4; b < kSteps / 4; ++b) {
            const float4 t = *reinterpret_cast<const float4*>(Lt + I * kSteps + 4 * b);
            if (4 * b > I) q[4 * b] = fmaf(-t.x, q[I], q[4 * b]);
            if (4 * b + 1 > I) q[4 * b + 1] = fmaf(-t.y, q[I], q[4 * b + 1]);
            if (4 * b + 2 > I) q[4 * b + 2] = fmaf(-t.z, q[I], q[4 * b + 2]);
            q[4 * b + 3] = fmaf(-t.w, q[I], q[4 * b + 3]);
        }
        Q[(size_t)I * nrowp] = q[I];
    }
    if constexpr (I + 1 < kSteps) solve_step<I + 1>(q, s, Lt, inv, Q, nrowp);
}

// NRL: rows a lane (nrow <= 32 NRL); phase D takes 32 / NRL candidates at a time.
template <int NRL>
__global__ void __launch_bounds__(kThreads, 1)
    rounds_kernel(int nrow, int ncol, const float* __restrict__ V, int npiv, Buf B, int* __restrict__ piv, unsigned* bar,
                  unsigned long long limit_ns) {
    extern __shared__ float4 smem_v4[];
    float* smem = reinterpret_cast<float*>(smem_v4);
    __shared__ int abort_sh, sh_min;
    __shared__ unsigned sh_hist[kBins], sh_u[kWarps];
    __shared__ unsigned long long sh_key[2][kWarps];
    __shared__ int sh_slot[2][kWarps], sh_piv[kSteps];
    __shared__ float red[kThreads], sh_inv[kSteps];
    unsigned gen = 0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nrowp = padded_rows(nrow);
    const int tiles = (ncol + kTile - 1) / kTile;
    const bool vec = ncol % 4 == 0 && reinterpret_cast<uintptr_t>(V) % 16 == 0;
    int k = 0;
    for (int round = 0; k < npiv; ++round) {
        const int par = round & 1;
        // ---- A: norms
        unsigned best = 0;
        if (round == 0) {
            for (int c = blockIdx.x * kThreads + tid; c < ncol; c += gridDim.x * kThreads) {
                float n0 = 0.f, n1 = 0.f, n2 = 0.f, n3 = 0.f;
                int r = 0;
#pragma unroll 4
                for (; r + 4 <= nrow; r += 4) {
                    const float a = __ldg(V + (size_t)r * ncol + c), e = __ldg(V + (size_t)(r + 1) * ncol + c);
                    const float f = __ldg(V + (size_t)(r + 2) * ncol + c), h = __ldg(V + (size_t)(r + 3) * ncol + c);
                    n0 += a * a;
                    n1 += e * e;
                    n2 += f * f;
                    n3 += h * h;
                }
                for (; r < nrow; ++r) {
                    const float a = __ldg(V + (size_t)r * ncol + c);
                    n0 += a * a;
                }
                const double n = (double)((n0 + n1) + (n2 + n3));
                __stcg(B.nrm + c, n);
                if (n >= 0.0) best = max(best, fbits(n));
            }
        } else {
            for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
                const float drop = norm_drop(V, nrow, ncol, B, t * kTile, vec, smem, red);
                const int c = t * kTile + tid;
                if (tid < kTile && c < ncol) {
                    double n = ld_nrm(B.nrm + c);
                    if (n >= 0.0) {
                        n = fmax(n - (double)drop, 0.0);
                        __stcg(B.nrm + c, n);
                        best = max(best, fbits(n));
                    }
                }
                __syncthreads();  // the stages are refilled
            }
        }
        best = __reduce_max_sync(0xffffffffu, best);
        if (lane == 0 && best) atomicMax(B.ctl + par, best);
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        const unsigned mkey = __ldcg(B.ctl + par);
        const float M = __uint_as_float(mkey), lo = 0.25f * M;
        // ---- B: histogram of the norms from lo to M
        for (int b = tid; b < kBins; b += kThreads) sh_hist[b] = 0;
        __syncthreads();
        for (int c = blockIdx.x * kThreads + tid; c < ncol; c += gridDim.x * kThreads) {
            const double n = ld_nrm(B.nrm + c);
            if (n >= 0.0 && (float)n >= lo) atomicAdd(&sh_hist[min((mkey - fbits(n)) >> 14, (unsigned)(kBins - 1))], 1u);
        }
        __syncthreads();
        for (int b = tid; b < kBins; b += kThreads)
            if (sh_hist[b]) atomicAdd(B.hist + b, sh_hist[b]);
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        // ---- C: bins 0 .. T-1 hold at most kCand columns; the others are at most tau
        {
            const unsigned a = __ldcg(B.hist + 2 * tid), e = __ldcg(B.hist + 2 * tid + 1);
            unsigned s = a + e;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += t;
            }
            if (lane == 31) sh_u[warp] = s;
            if (tid == 0) sh_min = kBins;
            __syncthreads();
            for (int w = 0; w < warp; ++w) s += sh_u[w];  // columns in bins 0 .. 2 tid + 1
            if (s - e > kCand) atomicMin(&sh_min, 2 * tid);
            else if (s > kCand) atomicMin(&sh_min, 2 * tid + 1);
            __syncthreads();
        }
        const int T = sh_min;
        const bool single = T == 0;  // more near-ties than candidates: take the largest norm alone
        const float tau = T >= kBins ? lo : fmaxf(__uint_as_float(mkey - min((unsigned)T << 14, mkey)), lo);
        for (int c = blockIdx.x * kThreads + tid; c < ncol; c += gridDim.x * kThreads) {
            const double n = ld_nrm(B.nrm + c);
            if (!(n >= 0.0) || (float)n < lo) continue;
            const unsigned key = fbits(n);
            if (single) {
                if (key == mkey) atomicMin(B.ctl + 4 + par, (unsigned)c);
            } else if ((int)((mkey - key) >> 14) < T) {
                const unsigned slot = atomicAdd(B.ctl + 2 + par, 1u);
                if (slot < kCand) __stcg(B.cand + slot, c);
            }
        }
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        const int cm = single ? 1 : (int)min(__ldcg(B.ctl + 2 + par), (unsigned)kCand);
        // ---- D: residuals of the candidates against every direction: each warp
        // takes every 16th direction for a few candidates at once
        {
            constexpr int CG = 32 / NRL;
            for (int m0 = blockIdx.x * CG; m0 < cm; m0 += gridDim.x * CG) {
                float v[CG][NRL], r[CG][NRL];
#pragma unroll
                for (int g = 0; g < CG; ++g) {
                    const int m = min(m0 + g, cm - 1);
                    const int c = single ? (int)__ldcg(B.ctl + 4 + par) : __ldcg(B.cand + m);
#pragma unroll
                    for (int i = 0; i < NRL; ++i) {
                        const int row = lane + 32 * i;
                        v[g][i] = row < nrow ? __ldg(V + (size_t)row * ncol + c) : 0.f;
                        r[g][i] = warp == 0 ? v[g][i] : 0.f;
                    }
                }
                for (int q = warp; q < k; q += kWarps) {
                    const float* qp = B.Q + (size_t)q * nrowp + lane;
                    float w[NRL], d[CG];
#pragma unroll
                    for (int i = 0; i < NRL; ++i) w[i] = lane + 32 * i < nrowp ? qp[32 * i] : 0.f;
#pragma unroll
                    for (int g = 0; g < CG; ++g) {
                        d[g] = 0.f;
#pragma unroll
                        for (int i = 0; i < NRL; ++i) d[g] = fmaf(w[i], v[g][i], d[g]);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                        for (int g = 0; g < CG; ++g) d[g] += __shfl_xor_sync(0xffffffffu, d[g], o);
#pragma unroll
                    for (int g = 0; g < CG; ++g)
#pragma unroll
                        for (int i = 0; i < NRL; ++i) r[g][i] = fmaf(-d[g], w[i], r[g][i]);
                }
                __syncthreads();
#pragma unroll
                for (int g = 0; g < CG; ++g)
#pragma unroll
                    for (int i = 0; i < NRL; ++i) smem[(warp * CG + g) * (32 * NRL) + lane + 32 * i] = r[g][i];
                __syncthreads();
                for (int e = tid; e < CG * 32 * NRL; e += kThreads) {
                    const int g = e / (32 * NRL), row = e % (32 * NRL);
                    float s = 0.f;
#pragma unroll
                    for (int w = 0; w < kWarps; ++w) s += smem[(w * CG + g) * (32 * NRL) + row];
                    if (m0 + g < cm && row < nrowp) __stcg(B.R + (size_t)(m0 + g) * nrowp + row, s);
                }
                if (single && tid == 0) __stcg(B.cand, (int)__ldcg(B.ctl + 4 + par));
            }
        }
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        // ---- E: their Gram matrix, 32 x 32 blocks on and above the diagonal
        {
            const int nb = (cm + 31) / 32, np = nb * (nb + 1) / 2;
            constexpr int P = 256 + 4;
            float* As = smem;
            float* Bs = smem + 32 * P;
            for (int t = blockIdx.x; t < np; t += gridDim.x) {
                int bi = 0, left = t;
                while (left >= nb - bi) {
                    left -= nb - bi;
                    ++bi;
                }
                const int bj = bi + left;
                const int i = tid >> 4, j = tid & 15;
                float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
                for (int r0 = 0; r0 < nrow; r0 += 256) {
                    const int len = min(256, nrowp - r0);
                    __syncthreads();
                    for (int e = tid; e < 32 * (len / 4); e += kThreads) {
                        const int row = e / (len / 4), q = e - row * (len / 4);
                        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                        const int ma = bi * 32 + row, mb = bj * 32 + row;
                        *reinterpret_cast<float4*>(As + row * P + 4 * q) =
                            ma < cm ? __ldcg(reinterpret_cast<const float4*>(B.R + (size_t)ma * nrowp + r0) + q) : z;
                        *reinterpret_cast<float4*>(Bs + row * P + 4 * q) =
                            mb < cm ? __ldcg(reinterpret_cast<const float4*>(B.R + (size_t)mb * nrowp + r0) + q) : z;
                    }
                    __syncthreads();
#pragma unroll 4
                    for (int q = 0; q < len; q += 4) {
                        const float4 a = *reinterpret_cast<const float4*>(As + i * P + q);
                        const float4 b = *reinterpret_cast<const float4*>(Bs + j * P + q);
                        const float4 e = *reinterpret_cast<const float4*>(Bs + (j + 16) * P + q);
                        s0.x = fmaf(a.x, b.x, s0.x);
                        s0.y = fmaf(a.y, b.y, s0.y);
                        s0.z = fmaf(a.z, b.z, s0.z);
                        s0.w = fmaf(a.w, b.w, s0.w);
                        s1.x = fmaf(a.x, e.x, s1.x);
                        s1.y = fmaf(a.y, e.y, s1.y);
                        s1.z = fmaf(a.z, e.z, s1.z);
                        s1.w = fmaf(a.w, e.w, s1.w);
                    }
                }
                const int m = bi * 32 + i, n0 = bj * 32 + j, n1 = n0 + 16;
                const float g0 = (s0.x + s0.y) + (s0.z + s0.w), g1 = (s1.x + s1.y) + (s1.z + s1.w);
                __stcg(B.G + (size_t)m * kCand + n0, g0);
                __stcg(B.G + (size_t)n0 * kCand + m, g0);
                __stcg(B.G + (size_t)m * kCand + n1, g1);
                __stcg(B.G + (size_t)n1 * kCand + m, g1);
            }
        }
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        // ---- F: pivots among the candidates
        if (blockIdx.x == 0) {
            float* Ls = smem;                     // [kCand][kLPitch] factor rows
            float* Lb = Ls + kCand * kLPitch;     // [8][kCand] entries of the steps of this block of eight
            float* Lt = Lb + 8 * kCand;           // [kSteps][kSteps]: the pivots' rows, transposed
            const int col = tid < cm ? __ldcg(B.cand + tid) : 0x7fffffff;
            float d = tid < cm ? fmaxf(__ldcg(B.G + (size_t)tid * kCand + tid), 0.f) : -1.f;
            const int most = min(single ? 1 : kSteps, npiv - k);
            float own[kSteps];  // this candidate's factor row, whole blocks of eight steps
#pragma unroll
            for (int l = 0; l < kSteps; ++l) own[l] = 0.f;
            int s = 0;
            for (;; ++s) {
                // largest residual norm, then lowest column
                const int hb = s & 1;
                {
                    const unsigned kh = d >= 0.f ? __float_as_uint(d) + 1u : 0u;
                    const unsigned hi = __reduce_max_sync(0xffffffffu, kh);
                    const unsigned lw = __reduce_max_sync(0xffffffffu, kh == hi ? ~(unsigned)col : 0u);
                    if (kh == hi && ~(unsigned)col == lw) {  // (idle slots of a warp write the same)
                        sh_key[hb][warp] = ((unsigned long long)hi << 32) | lw;
                        sh_slot[hb][warp] = tid;
                    }
                }
                __syncthreads();
                const unsigned long long w = lane < kWarps ? sh_key[hb][lane] : 0ull;
                const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(w >> 32));
                const unsigned lw = __reduce_max_sync(0xffffffffu, (unsigned)(w >> 32) == hi ? (unsigned)w : 0u);
                const float dmax = hi ? __uint_as_float(hi - 1u) : 0.f;
                // the first is the largest norm of all; the others have to stay above tau
                // (by more than the rounding of the norms outside)
                if (s == most || !hi || (s > 0 && !(dmax > tau * (1.f + 4e-6f)))) break;
                const unsigned who = __ballot_sync(0xffffffffu, lane < kWarps && w == (((unsigned long long)hi << 32) | lw));
                const int p = sh_slot[hb][__ffs(who) - 1];
                const float g = tid < cm ? __ldcg(B.G + (size_t)p * kCand + tid) : 0.f;
                // L_p . L_j over the earlier steps (summed while the Gram row is on its way)
                const float* lp = Ls + p * kLPitch;
                float a0 = 0.f, a1 = 0.f;
#pragma unroll
                for (int b = 0; b < kSteps / 8; ++b) {
                    if (8 * b + 8 <= s) {
                        const float4 x = *reinterpret_cast<const float4*>(lp + 8 * b), y = *reinterpret_cast<const float4*>(lp + 8 * b + 4);
                        a0 = fmaf(x.x, own[8 * b], a0);
                        a1 = fmaf(x.y, own[8 * b + 1], a1);
                        a0 = fmaf(x.z, own[8 * b + 2], a0);
                        a1 = fmaf(x.w, own[8 * b + 3], a1);
                        a0 = fmaf(y.x, own[8 * b + 4], a0);
                        a1 = fmaf(y.y, own[8 * b + 5], a1);
                        a0 = fmaf(y.z, own[8 * b + 6], a0);
                        a1 = fmaf(y.w, own[8 * b + 7], a1);
                    }
                }
                for (int l = s & ~7; l < s; ++l) a0 = fmaf(lp[l], Lb[(l & 7) * kCand + tid], a0);
                const float root = sqrtf(dmax), inv = dmax > 0.f ? 1.f / root : 0.f;
                const float x = tid == p ? root : (g - (a0 + a1)) * inv;
                Ls[tid * kLPitch + s] = x;
                Lb[(s & 7) * kCand + tid] = x;
                if (tid == p) {
                    d = -1.f;
                    sh_piv[s] = p;
                    sh_inv[s] = inv;
                    piv[k + s] = col;
                    __stcg(B.nrm + col, -1.0);
                } else if (d >= 0.f) {
                    d = fmaxf(fmaf(-x, x, d), 0.f);
                }
                if ((s & 7) == 7) {
#pragma unroll
                    for (int l = 0; l < 8; ++l) {
                        const float e = Lb[l * kCand + tid];
#pragma unroll
                        for (int b = 0; b < kSteps / 8; ++b) own[8 * b + l] = b == s >> 3 ? e : own[8 * b + l];
                    }
                }
            }
            __syncthreads();
            for (int e = tid; e < kSteps * kSteps; e += kThreads) {
                const int i = e / kSteps, l = e % kSteps;  // Lt[i][l] = L[pivot l][step i], l > i
                Lt[e] = i < s && l < s && l > i ? Ls[sh_piv[l] * kLPitch + i] : 0.f;
            }
            __syncthreads();
            // directions: q_i = (r_i - sum_{l < i} L_il q_l) / L_ii, a row of the
            // pivots' residuals a thread
            for (int row = tid; row < nrowp; row += kThreads) {
                float q[kSteps];
#pragma unroll
                for (int i = 0; i < kSteps; ++i) q[i] = i < s ? __ldcg(B.R + (size_t)sh_piv[i] * nrowp + row) : 0.f;
                solve_step<0>(q, s, Lt, sh_inv, B.Q + (size_t)k * nrowp + row, nrowp);
                float4* o = reinterpret_cast<float4*>(B.QT + (size_t)row * kSteps);
#pragma unroll
                for (int i = 0; i < kSteps / 4; ++i) o[i] = make_float4(q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);
            }
            if (s == 0) {
                // no norm compares (NaN input): any columns, so that the launch ends
                if (tid == 0) {
                    int c = 0;
                    for (int i = k; i < npiv; ++i) {
                        while (ld_nrm(B.nrm + c) == -1.0) ++c;
                        piv[i] = c;
                        __stcg(B.nrm + c, -1.0);
                    }
                }
                s = npiv - k;
            }
            // the next round's counters
            for (int b = tid; b < kBins; b += kThreads) B.hist[b] = 0;
            if (tid == 0) {
                B.ctl[par ^ 1] = 0;
                B.ctl[2 + (par ^ 1)] = 0;
                B.ctl[4 + (par ^ 1)] = 0xffffffffu;
                B.ctl[6] = k + s;
            }
        }
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        k = (int)__ldcg(B.ctl + 6);
    }
}

}  // namespace qrr
}  // namespace lace
