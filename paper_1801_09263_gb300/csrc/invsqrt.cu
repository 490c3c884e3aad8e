// Inverse square roots of symmetric positive definite N x N matrices (Loewdin
// orthonormalisation, the SCDM rotation and the alignment, Sec. 2) by the
// coupled Newton-Schulz iteration (Higham, "Functions of Matrices", Sec. 6.7):
//   Y_0 = A/c, Z_0 = I;  T = (3 I - Z Y)/2;  Y <- Y T,  Z <- T Z;  Z -> (A/c)^{-1/2}
// with c = ||A||_inf >= lambda_max, so that the spectrum starts in (0, 1].
//
// One launch runs the whole iteration, its convergence test included: the
// products are small (33 MFLOP at N = 256) and the launches, the elementwise
// kernels between them and the host's waits for the norms were most of the time.
// Up to 16 rows one CTA keeps everything in shared memory, up to 64 in FP32 a
// cluster of eight does; beyond, a cooperative grid computes tiles and meets at a
// barrier after every product.  The iterates are symmetric but for rounding, and yet all products
// are computed whole and read as they stand: the iteration damps the errors of
// Z Y, Y T and T Z alone.  With T mirrored from its upper triangle they grow by
// sqrt(lambda_max / lambda_min) a step (FP32 X A X - I of 2e-2 instead of 6e-5 at N = 400
// and 2.5e3); with Y and Z mirrored, or a transpose read in place of either, matrices of
// 1e7 that converge do not.
//
// Measured (FP32, both inverse square roots of a step, kernels alone): 364 us at
// N = 256 and 114 us at N = 64; separate launches with their waits took 650 and 480 us.
#include <algorithm>
#include <cmath>

#include "cta_sums.cuh"
#include "grid_sync.cuh"
#include "lace_internal.cuh"

namespace lace {
namespace {

constexpr int kNsThreads = 256;
constexpr int kNsMaxIt = 160;
constexpr int kNsMaxCtas = 304;

// Convergence of h = ||I - Z Y||_F^2 = sum (1 - x_k)^2 over the eigenvalues of
// Z Y.  FP64: once below 1e-24 N this step is the last, for the bound leaves |1 - x_k| at
// up to 1e-12 and a step squares it to the rounding level (without it FP64 orbitals
// of 48^3 x 32 were off by 4e-14 instead of 4e-15); or below 1e-12 N and no longer falling
// by 4x (the rounding floor) without another.  FP32: below 1e-11 N, or the same floor
// below 1e-6 N; and once below 1e-6 N
// every |1 - x_k| < 0.016 and the iteration is in its quadratic regime
// (1 - x -> ~(3/4)(1 - x)^2), so two more steps reach the floor.
// h is summed in FP32 (FP64 runs at 1/64 of its rate, and a sum of the squares of
// FP64 differences needs neither its digits nor its range).
template <typename T> struct Stop {
    float prev;
    int extra;  // steps left after this one, once they are counted
    __device__ Stop() : prev(INFINITY), extra(-1) {}
    // the last step is done
    __device__ bool done() const { return extra == 0; }
    // 1: converged, 0: go on, -1: failed
    __device__ int test(float h, int n) {
        constexpr float lo = sizeof(T) == 8 ? 1e-24f : 1e-11f, hi = sizeof(T) == 8 ? 1e-12f : 1e-6f;
        if (extra > 0) {
            --extra;
            return 0;
        }
        if (!(h < INFINITY)) return -1;
        if (h < lo * n) {
            if (sizeof(T) == 4) return 1;
            extra = 0;
            return 0;
        }
        if (h < hi * n && h > 0.25f * prev) return 1;
        if (sizeof(T) == 4 && h < hi * n) extra = 1;  // this step and one more
        prev = h;
        return 0;
    }
};

template <typename V> __device__ __forceinline__ V block_sum(V v, V* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    V t = V(0);
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    return t;
}

// ------------------------------------------------------------------ one CTA
// NB consecutive values.
template <typename T, int NB> __device__ __forceinline__ void load_row(const T* p, T* v) {
    if constexpr (sizeof(T) == 4 && NB == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else if constexpr (sizeof(T) == 4 && NB == 2) {
        const float2 q = *reinterpret_cast<const float2*>(p);
        v[0] = q.x, v[1] = q.y;
    } else {
#pragma unroll
        for (int j = 0; j < NB; ++j) v[j] = p[j];
    }
}

// C = A B of matrices in shared memory (16 rows of pitch P, zero past N), one
// output a thread; f(m, n, value) for every output.
template <typename T, int P, class F> __device__ __forceinline__ void one_product(int N, const T* A, const T* B, F f) {
    const int m = threadIdx.x >> 4, n = threadIdx.x & 15;
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fma(A[m * P + k], B[k * P + n], acc);
    if (m < N && n < N) f(m, n, acc);
}

template <typename T>
__global__ void __launch_bounds__(kNsThreads) ns_one_kernel(int N, const double* __restrict__ A, double* __restrict__ X,
                                                            int* status) {
    constexpr int R = 16, P = 17;
    __shared__ T mats[5 * R * P];
    __shared__ double sh[kNsThreads / 32];
    __shared__ float shf[kNsThreads / 32];
    T* Y = mats;
    T* Z = Y + R * P;
    T* W = Z + R * P;
    T* Y2 = W + R * P;
    T* Z2 = Y2 + R * P;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // c = largest row sum
    double c = 0.0;
    for (int r = warp; r < N; r += kNsThreads / 32) {
        double s = 0.0;
        for (int k = lane; k < N; k += 32) s += fabs(A[(size_t)r * N + k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        c = s > c || s != s ? s : c;
    }
    if (lane == 0) sh[warp] = c;
    __syncthreads();
    c = 0.0;
    for (int w = 0; w < kNsThreads / 32; ++w) c = sh[w] > c || sh[w] != sh[w] ? sh[w] : c;
    if (tid == 0) *status = 0;
    if (!(c > 0.0) || !(c < INFINITY)) return;
    const double ci = 1.0 / c;
    for (int e = tid; e < 5 * R * P; e += kNsThreads) Y[e] = T(0);
    __syncthreads();
    for (int e = tid; e < N * N; e += kNsThreads) {
        const int r = e / N, k = e % N;
        Y[r * P + k] = (T)(0.5 * (A[e] + A[(size_t)k * N + r]) * ci);
        if (r == k) Z[r * P + k] = T(1);
    }
    __syncthreads();
    Stop<T> stop;
    bool ok = false;
    for (int it = 0; it < kNsMaxIt; ++it) {
        if (stop.done()) {
            ok = true;
            break;
        }
        float h = 0.f;
        one_product<T, P>(N, Z, Y, [&](int m, int n, T v) {
            const T d = m == n ? T(1) : T(0);
            const float x = (float)(d - v);
            h = fmaf(x, x, h);
            W[m * P + n] = T(0.5) * (T(2) * d + (d - v));  // (3 delta - v) / 2
        });
        h = block_sum(h, shf);
        const int st = stop.test(h, N);
        if (st != 0) {
            ok = st > 0;
            break;
        }
        one_product<T, P>(N, Y, W, [&](int m, int n, T v) { Y2[m * P + n] = v; });
        one_product<T, P>(N, W, Z, [&](int m, int n, T v) { Z2[m * P + n] = v; });
        __syncthreads();
        T* t = Y;
        Y = Y2;
        Y2 = t;
        t = Z;
        Z = Z2;
        Z2 = t;
    }
    // ||(A/c)^{-1/2}||_F^2 >= lambda_max / lambda_min: reject ill-conditioned A
    double f = 0.0;
    for (int e = tid; e < N * N; e += kNsThreads) {
        const double z = 0.5 * ((double)Z[(e / N) * P + e % N] + (double)Z[(e % N) * P + e / N]);
        f += z * z;
    }
    f = block_sum(f, sh);
    if (!ok || !(f < 1e12)) return;
    const double s = 1.0 / sqrt(c);
    for (int e = tid; e < N * N; e += kNsThreads) 
        X[e] = s * 0.5 * ((double)Z[(e / N) * P + e % N] + (double)Z[(e % N) * P + e / N]);
    if (tid == 0) *status = 1;
}

// ------------------------------------------------------------------ a cluster
// 17 to 64 rows in FP32: eight CTAs with a copy of the iterates each compute
// RB rows of a product and write them into all copies (distributed shared
// memory); two cluster barriers a step.  One CTA took 139 us for a 64 x 64 of a 48^3
// step (3.2 us a step at the FP32 peak of one SM), this takes 57: load and
// localisation 0.71 -> 0.54 ms.  At 80 and 96 rows it is even with the grid (0.15 and
// 0.16 ms a load).
constexpr int kNsCluster = 8;
template <int RB> struct NsCl {
    static constexpr int R = kNsCluster * RB, P = R + 4;
    static constexpr int KG = RB == 4 ? 8 : 4;  // groups of threads, each a part of K
    static constexpr int UNITS = RB * RB, THREADS = UNITS * KG;  // 4 rows x 2 columns a thread
    static constexpr int FLOATS = 4 * R * P + 2 * KG * RB * R;
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The shared-memory address of p in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}

// Partial sums over this group's part of K of RB rows of A B -> red[group].
template <int RB> __device__ __forceinline__ void cl_product(const float* A, const float* B, float* red) {
    using C = NsCl<RB>;
    const int group = threadIdx.x / C::UNITS, u = threadIdx.x % C::UNITS;
    const int r0 = u / (C::R / 2) * 4, c0 = u % (C::R / 2) * 2;
    float acc[4][2] = {};
#pragma unroll 4
    for (int k = group * (C::R / C::KG); k < (group + 1) * (C::R / C::KG); k += 4) {
        float a[4][4], b[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) load_row<float, 4>(A + (r0 + i) * C::P + k, a[i]);
#pragma unroll
        for (int q = 0; q < 4; ++q) load_row<float, 2>(B + (k + q) * C::P + c0, b[q]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) acc[i][j] = fmaf(a[i][q], b[q][j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float2*>(red + (group * RB + r0 + i) * C::R + c0) = make_float2(acc[i][0], acc[i][1]);
}
// Four outputs of a row (e = 4-column group of RB x R) summed over the groups.
template <int RB> __device__ __forceinline__ float4 cl_sum(const float* red, int e) {
    using C = NsCl<RB>;
    float4 s = *reinterpret_cast<const float4*>(red + 4 * e);
#pragma unroll
    for (int g = 1; g < C::KG; ++g) {
        const float4 v = *reinterpret_cast<const float4*>(red + g * RB * C::R + 4 * e);
        s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
    }
    return s;
}
__device__ __forceinline__ void cl_put(float* at, float4 v) {
#pragma unroll
    for (int r = 0; r < kNsCluster; ++r)
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(cluster_addr(at, r)), "f"(v.x), "f"(v.y), "f"(v.z),
                     "f"(v.w)
                     : "memory");
}

template <int RB>
__global__ void __cluster_dims__(kNsCluster, 1, 1) __launch_bounds__(NsCl<RB>::THREADS)
    ns_cluster_kernel(int N, const double* __restrict__ A, double* __restrict__ X, int* status) {
    using C = NsCl<RB>;
    constexpr int R = C::R, P = C::P, TH = C::THREADS;
    extern __shared__ double ns_smem[];
    __shared__ float sh[TH / 32 + 1];
    __shared__ float part[kNsCluster];
    __shared__ double rowsum[TH / 32 + 1];
    float* Y = reinterpret_cast<float*>(ns_smem);
    float* Z = Y + R * P;
    float* Z2 = Z + R * P;
    float* W = Z2 + R * P;
    float* red = W + R * P;
    float* red2 = red + C::KG * RB * R;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = (int)cluster_rank(), m0 = rank * RB;
    // c = largest row sum (every CTA for itself)
    double c = 0.0;
    for (int r = warp; r < N; r += TH / 32) {
        double s = 0.0;
        for (int k = lane; k < N; k += 32) s += fabs(A[(size_t)r * N + k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        c = s > c || s != s ? s : c;
    }
    if (lane == 0) rowsum[warp] = c;
    __syncthreads();
    c = 0.0;
    for (int w = 0; w < TH / 32; ++w) c = rowsum[w] > c || rowsum[w] != rowsum[w] ? rowsum[w] : c;
    const bool run = c > 0.0 && c < INFINITY;  // (alike in all CTAs)
    const double ci = run ? 1.0 / c : 0.0;
    for (int e = tid; e < 3 * R * P; e += TH) Y[e] = 0.f;
    __syncthreads();
    for (int e = tid; e < N * N; e += TH) {
        const int r = e / N, k = e % N;
        Y[r * P + k] = (float)(0.5 * (A[e] + A[(size_t)k * N + r]) * ci);
        if (r == k) Z[r * P + k] = 1.f;
    }
    cluster_barrier();  // all copies are set up
    Stop<float> stop;
    bool ok = false;
    if (run)
        for (int it = 0; it < kNsMaxIt; ++it) {
            if (stop.done()) {
                ok = true;
                break;
            }
            cl_product<RB>(Z + m0 * P, Y, red);
            __syncthreads();
            float h = 0.f;
            for (int e = tid; e < RB * R / 4; e += TH) {
                const int m = m0 + 4 * e / R, n = 4 * e % R;
                const float4 v = cl_sum<RB>(red, e);
                float4 t;
                auto one = [&](float v1, int col) {
                    const float d = m == col ? 1.f : 0.f, x = m < N && col < N ? d - v1 : 0.f;
                    h = fmaf(x, x, h);
                    return m < N && col < N ? 0.5f * (2.f * d + x) : 0.f;  // (3 delta - v) / 2
                };
                t.x = one(v.x, n), t.y = one(v.y, n + 1), t.z = one(v.z, n + 2), t.w = one(v.w, n + 3);
                cl_put(W + m * P + n, t);
            }
            h = block_sum(h, sh);
            if (tid < kNsCluster)
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(part + rank, tid)), "f"(h) : "memory");
            cluster_barrier();
            h = 0.f;
#pragma unroll
            for (int r = 0; r < kNsCluster; ++r) h += part[r];  // a fixed order: every CTA decides alike
            const int st = stop.test(h, N);
            if (st != 0) {
                ok = st > 0;
                break;
            }
            cl_product<RB>(Y + m0 * P, W, red);
            cl_product<RB>(W + m0 * P, Z, red2);
            __syncthreads();  // (Y's own rows are read: the other CTAs read no rows of this one's now)
            for (int e = tid; e < RB * R / 4; e += TH) {
                const int at = (m0 + 4 * e / R) * P + 4 * e % R;
                cl_put(Y + at, cl_sum<RB>(red, e));
                cl_put(Z2 + at, cl_sum<RB>(red2, e));
            }
            cluster_barrier();
            float* t = Z;
            Z = Z2;
            Z2 = t;
        }
    // ||(A/c)^{-1/2}||_F^2 >= lambda_max / lambda_min: reject ill-conditioned A
    float f = 0.f;
    const double s = 1.0 / sqrt(c);
    for (int e = tid; e < N * N; e += TH) {
        const float z = 0.5f * (Z[(e / N) * P + e % N] + Z[(e % N) * P + e / N]);
        f = fmaf(z, z, f);
    }
    f = block_sum(f, sh);
    ok = ok && f < 1e12f;
    if (ok)
        for (int e = rank * TH + tid; e < N * N; e += kNsCluster * TH)
            X[e] = s * 0.5 * ((double)Z[(e / N) * P + e % N] + (double)Z[(e % N) * P + e / N]);
    if (rank == 0 && tid == 0) *status = ok ? 1 : 0;
    cluster_barrier();  // no CTA leaves while its memory may be written
}

// ------------------------------------------------------------------ a grid
// Tile sizes: FP32 16 x 16 outputs, 2 x 2 a thread; FP64 8 x 8, one a thread.
// Four groups of 64 threads take a quarter of K each.
template <typename T> struct NsTile;
template <> struct NsTile<float> {
    static constexpr int S = 16, KC = 256, P = KC + 4, E = 2;
};
template <> struct NsTile<double> {
    static constexpr int S = 8, KC = 128, P = KC + 1, E = 1;
};

template <typename T> struct NsArgs {
    int N, ld;
    const double* A;
    double* X;
    T *Y, *Z, *W, *Y2, *Z2;    // N rows of ld
    float* part;               // CtaSums::kRows x kNsMaxCtas
    unsigned* bar;             // 4, zero at launch
    unsigned long long* norm;  // zero at launch
    unsigned long long limit_ns;  // of a barrier wait
    int* status;               // 1 converged, 0 failed, -1 a barrier wait ran out (preset)
};

// One tile (bm, bn) of A B; f(m, n, value) for its outputs, each by one thread.
template <typename T, class F>
__device__ __forceinline__ void grid_product(int N, int ld, const T* A, const T* B, int bm, int bn, T* smem, F f) {
    using C = NsTile<T>;
    constexpr int S = C::S, P = C::P, E = C::E, KV = sizeof(T) == 4 ? 4 : 1;
    T* As = smem;          // [S][P]
    T* Bs = smem + S * P;  // [KC][S]
    T* red = Bs + C::KC * S;  // [4][S][S]
    const int tid = threadIdx.x, group = tid >> 6, t = tid & 63, ti = t >> 3, tj = t & 7;
    T acc[E][E];
#pragma unroll
    for (int i = 0; i < E; ++i)
#pragma unroll
        for (int j = 0; j < E; ++j) acc[i][j] = T(0);
    for (int k0 = 0; k0 < N; k0 += C::KC) {
        const int len = min(C::KC, N - k0), per = ((len + 3) / 4 + 3) / 4 * 4;  // (past len: zeros)
        __syncthreads();
        if constexpr (sizeof(T) == 4) {
            constexpr int Q = C::KC / 4, SQ = S / 4;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int e = tid; e < S * Q; e += kNsThreads) {
                const int r = e / Q, q = e % Q, row = bm * S + r;
                *reinterpret_cast<float4*>(As + r * P + 4 * q) =
                    row < N && k0 + 4 * q < ld ? __ldcg(reinterpret_cast<const float4*>(A + (size_t)row * ld + k0) + q) : z;
            }
            for (int e = tid; e < 4 * per * SQ; e += kNsThreads) {
                const int k = e / SQ, q = e % SQ, col = bn * S + 4 * q;
                *reinterpret_cast<float4*>(Bs + k * S + 4 * q) =
                    k < len && col < ld ? __ldcg(reinterpret_cast<const float4*>(B + (size_t)(k0 + k) * ld + col)) : z;
            }
        } else {
            for (int e = tid; e < S * C::KC; e += kNsThreads) {
                const int r = e / C::KC, q = e % C::KC, row = bm * S + r;
                As[r * P + q] = row < N && q < len ? __ldcg(A + (size_t)row * ld + k0 + q) : T(0);
            }
            for (int e = tid; e < S * C::KC; e += kNsThreads) {
                const int k = e / S, col = bn * S + e % S;
                Bs[e] = k < len && col < N ? __ldcg(B + (size_t)(k0 + k) * ld + col) : T(0);
            }
        }
        __syncthreads();
        const int kb = group * per, ke = min(kb + per, C::KC);
        for (int k = kb; k < ke; k += KV) {
            T a[E][KV], b[KV][E];
#pragma unroll
            for (int i = 0; i < E; ++i) load_row<T, KV>(As + (ti + 8 * i) * P + k, a[i]);
#pragma unroll
            for (int q = 0; q < KV; ++q) load_row<T, E>(Bs + (k + q) * S + E * tj, b[q]);
#pragma unroll
            for (int q = 0; q < KV; ++q)
#pragma unroll
                for (int i = 0; i < E; ++i)
#pragma unroll
                    for (int j = 0; j < E; ++j) acc[i][j] = fma(a[i][q], b[q][j], acc[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < E; ++i)
#pragma unroll
        for (int j = 0; j < E; ++j) red[(group * S + ti + 8 * i) * S + E * tj + j] = acc[i][j];
    __syncthreads();
    if (tid < S * S) {
        const int m = bm * S + tid / S, n = bn * S + tid % S;
        const T v = (red[tid] + red[S * S + tid]) + (red[2 * S * S + tid] + red[3 * S * S + tid]);
        if (m < N && n < N) f(m, n, v);
    }
    __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kNsThreads) ns_grid_kernel(NsArgs<T> a) {
    using C = NsTile<T>;
    __shared__ __align__(16) T smem[C::S * (C::P + C::KC) + 4 * C::S * C::S];
    __shared__ float sh[kNsThreads / 32];
    __shared__ int abort_sh;
    unsigned gen = 0;
    const int N = a.N, ld = a.ld, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nt = (N + C::S - 1) / C::S, tiles = nt * nt;
    const size_t all = (size_t)gridDim.x * kNsThreads, me = (size_t)blockIdx.x * kNsThreads + tid;
    // c = largest row sum
    for (int r = blockIdx.x * (kNsThreads / 32) + warp; r < N; r += gridDim.x * (kNsThreads / 32)) {
        double s = 0.0;
        for (int k = lane; k < N; k += 32) s += fabs(__ldg(a.A + (size_t)r * N + k));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) atomicMax(a.norm, (unsigned long long)__double_as_longlong(s));  // (a NaN is the largest)
    }
    if (!grid_barrier(a.bar, gen, &abort_sh, a.limit_ns)) return;
    const double c = __longlong_as_double((long long)__ldcg(a.norm));
    if (!(c > 0.0) || !(c < INFINITY)) {
        if (me == 0) *a.status = 0;
        return;
    }
    // the first step: Z = I, so T = (3 I - Y)/2 and Z_1 = T
    const double ci = 1.0 / c;
    for (size_t e = me; e < (size_t)N * ld; e += all) {
        const int r = (int)(e / ld), k = (int)(e % ld);
        T y = T(0), t = T(0);
        if (k < N) {
            y = (T)(0.5 * (__ldg(a.A + (size_t)r * N + k) + __ldg(a.A + (size_t)k * N + r)) * ci);
            t = T(0.5) * ((r == k ? T(3) : T(0)) - y);
        }
        __stcg(a.Y + e, y);
        __stcg(a.W + e, t);
        __stcg(a.Z2 + e, t);
        __stcg(a.Y2 + e, T(0));  // (the padding of the rows stays zero)
        __stcg(a.Z + e, T(0));
    }
    if (!grid_barrier(a.bar, gen, &abort_sh, a.limit_ns)) return;
    T *Y = a.Y, *Z = a.Z, *Y2 = a.Y2, *Z2 = a.Z2;
    auto put = [&](T* M, int m, int n, T v) { __stcg(M + (size_t)m * ld + n, v); };
    // v summed over the CTAs in a fixed order, so that every CTA decides alike; false: a
    // barrier wait ran out
    CtaSums sums;
    auto total = [&](float& v) {
        if (tid == 0) __stcg(a.part + sums.at(blockIdx.x, kNsMaxCtas), v);
        if (!grid_barrier(a.bar, gen, &abort_sh, a.limit_ns)) return false;
        float s = 0.f;
        if (warp == 0) {
            for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(a.part + sums.at(b, kNsMaxCtas));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) sh[0] = s;
        }
        __syncthreads();
        v = sh[0];
        __syncthreads();
        sums.next();
        return true;
    };
    Stop<T> stop;
    bool ok = false;
    for (int it = 0; it < kNsMaxIt; ++it) {
        if (stop.done()) {
            ok = true;
            break;
        }
        if (it > 0) {
            float h = 0.f;
            for (int t = blockIdx.x; t < tiles; t += gridDim.x)
                grid_product<T>(N, ld, Z, Y, t / nt, t % nt, smem, [&](int m, int n, T v) {
                    const T d = m == n ? T(1) : T(0);
                    const float x = (float)(d - v);
                    h = fmaf(x, x, h);
                    put(a.W, m, n, T(0.5) * (T(2) * d + (d - v)));
                });
            h = block_sum(h, sh);
            if (!total(h)) return;
            const int st = stop.test(h, N);
            if (st != 0) {
                ok = st > 0;
                break;
            }
        }
        for (int t = blockIdx.x; t < (it > 0 ? 2 : 1) * tiles; t += gridDim.x) {
            const int bm = t % tiles / nt, bn = t % nt;
            if (t < tiles) grid_product<T>(N, ld, Y, a.W, bm, bn, smem, [&](int m, int n, T v) { put(Y2, m, n, v); });
            else grid_product<T>(N, ld, a.W, Z, bm, bn, smem, [&](int m, int n, T v) { put(Z2, m, n, v); });
        }
        if (!grid_barrier(a.bar, gen, &abort_sh, a.limit_ns)) return;
        T* t = Y;
        Y = Y2;
        Y2 = t;
        t = Z;
        Z = Z2;
        Z2 = t;
    }
    // ||(A/c)^{-1/2}||_F^2 >= lambda_max / lambda_min: reject ill-conditioned A
    auto sym = [&](size_t e) {
        return 0.5 * ((double)__ldcg(Z + (e / N) * ld + e % N) + (double)__ldcg(Z + (e % N) * ld + e / N));
    };
    float f = 0.f;
    for (size_t e = me; e < (size_t)N * N; e += all) {
        const float z = (float)sym(e);
        f = fmaf(z, z, f);
    }
    f = block_sum(f, sh);
    if (!total(f)) return;
    ok = ok && f < 1e12f;
    const double s = 1.0 / sqrt(c);
    if (ok)
        for (size_t e = me; e < (size_t)N * N; e += all) a.X[e] = s * sym(e);
    // (a CTA whose wait for the sum ran out has not written its share)
    if (!grid_barrier(a.bar, gen, &abort_sh, a.limit_ns)) return;
    if (me == 0) *a.status = ok ? 1 : 0;
}

template <int RB> cudaError_t ns_cluster(int N, const double* A, double* X, int* d_status, cudaStream_t s) {
    using C = NsCl<RB>;
    constexpr size_t sm = C::FLOATS * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute((const void*)ns_cluster_kernel<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e) return e;
    ns_cluster_kernel<RB><<<kNsCluster, C::THREADS, sm, s>>>(N, A, X, d_status);
    return cudaGetLastError();
}

// X = A^{-1/2}; work: five N x ld matrices of T, then the control words.
template <typename T>
cudaError_t inv_sqrt(int N, const double* A, double* X, double* work, unsigned long long wait_limit_ns, int* d_status,
                     cudaStream_t s, int* launches) {
    const int ld = sizeof(T) == 4 ? (N + 3) / 4 * 4 : N;
    const size_t mat = ((size_t)N * ld * sizeof(T) + 15) / 16 * 16;
    unsigned char* w = reinterpret_cast<unsigned char*>(((uintptr_t)work + 15) & ~(uintptr_t)15);
    unsigned char* ctl = w + 5 * mat;
    cudaError_t e;
    const bool small = N <= (sizeof(T) == 4 ? 64 : 16);
    if (small) {
        if (N <= 16) {
            ns_one_kernel<T><<<1, kNsThreads, 0, s>>>(N, A, X, d_status);
            e = cudaGetLastError();
        } else if (N <= 32) e = ns_cluster<4>(N, A, X, d_status, s);
        else e = ns_cluster<8>(N, A, X, d_status, s);
        if (e) return e;
    } else {
        if ((e = cudaMemsetAsync(d_status, 0xff, sizeof(int), s))) return e;        // status -1
        if ((e = cudaMemsetAsync(ctl + 16, 0, 32, s))) return e;               // barrier, norm
        NsArgs<T> a;
        a.N = N;
        a.ld = ld;
        a.A = A;
        a.X = X;
        a.Y = reinterpret_cast<T*>(w);
        a.Z = reinterpret_cast<T*>(w + mat);
        a.W = reinterpret_cast<T*>(w + 2 * mat);
        a.Y2 = reinterpret_cast<T*>(w + 3 * mat);
        a.Z2 = reinterpret_cast<T*>(w + 4 * mat);
        a.status = d_status;
        a.bar = reinterpret_cast<unsigned*>(ctl + 16);
        a.norm = reinterpret_cast<unsigned long long*>(ctl + 32);
        a.limit_ns = wait_limit_ns;
        a.part = reinterpret_cast<float*>(ctl + 64);
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const void* fn = (const void*)ns_grid_kernel<T>;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kNsThreads, 0))) return e;
        if (per_sm < 1 || sms > kNsMaxCtas) return cudaErrorCooperativeLaunchTooLarge;
        const int nt = (N + NsTile<T>::S - 1) / NsTile<T>::S;
        // the two products of a step side by side
        const int ctas = std::min({sms * std::min(per_sm, 2), kNsMaxCtas, 2 * nt * nt});
        void* args[] = {(void*)&a};
        if ((e = cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(kNsThreads), args, 0, s))) return e;
    }
    *launches += 1;
    return cudaSuccess;
}

}  // namespace

cudaError_t inv_sqrt_spd(int N, const double* A, double* X, double* work, unsigned long long wait_limit_ns, int* d_status,
                         cudaStream_t s, int* launches) {
    return inv_sqrt<double>(N, A, X, work, wait_limit_ns, d_status, s, launches);
}
cudaError_t inv_sqrt_spd_mixed(int N, const double* A, double* X, double* work, unsigned long long wait_limit_ns,
                               int* d_status, cudaStream_t s, int* launches) {
    return inv_sqrt<float>(N, A, X, work, wait_limit_ns, d_status, s, launches);
}

}  // namespace lace
