// Inverse square roots of symmetric positive definite N x N matrices (Loewdin
// orthonormalisation, the SCDM rotation and the alignment, Sec. 2) by the
// coupled Newton-Schulz iteration (Higham, "Functions of Matrices", Sec. 6.7):
//   Y_0 = A/c, Z_0 = I;  T = (3 I - Z Y)/2;  Y <- Y T,  Z <- T Z;  Z -> (A/c)^{-1/2}
// with c = ||A||_inf >= lambda_max, so that the spectrum starts in (0, 1].
//
// One launch runs the whole iteration, its convergence test included: the
// products are small (33 MFLOP at N = 256) and the launches, the elementwise
// kernels between them and the host's waits for the norms were most of the time.
// Up to 64 rows in FP32 (16 in FP64) one CTA keeps everything in shared memory;
// beyond, a cooperative grid computes tiles and meets at a barrier after every
// product.  The iterates are symmetric but for rounding, and yet all products
// are computed whole and read as they stand: the iteration damps the errors of
// Z Y, Y T and T Z alone.  With T mirrored from its upper triangle they grow by
// sqrt(lambda_max / lambda_min) a step (FP32 X A X - I of 2e-2 instead of 6e-5 at N = 400
// and 2.5e3); with Y and Z mirrored, or a transpose read in place of either, matrices of
// 1e7 that converge do not.
//
// Measured (FP32, both inverse square roots of a step): kernels 2 x 226 us at
// N = 256 and 2 x 139 us at N = 64; separate launches with their waits took 650 and 480 us.
#include <algorithm>
#include <cmath>

#include "grid_sync.cuh"
#include "lace_internal.cuh"

namespace lace {
namespace {

constexpr int kNsThreads = 256;
constexpr int kNsMaxIt = 160;
constexpr int kNsMaxCtas = 304;

// Convergence of h = ||I - Z Y||_F^2 = sum (1 - x_k)^2 over the eigenvalues of
// Z Y.  FP64: below 1e-24 N, or below 1e-12 N and no longer falling by 4x (the
// rounding floor).  FP32: the same at 1e-11 N and 1e-6 N; and once below 1e-6 N
// every |1 - x_k| < 0.016 and the iteration is in its quadratic regime
// (1 - x -> ~(3/4)(1 - x)^2), so two more steps reach the floor.
template <typename T> struct Stop {
    double prev;
    int extra;
    __device__ Stop() : prev(INFINITY), extra(-1) {}
    // the last of the two extra steps is done
    __device__ bool done() const { return extra == 0; }
    // 1: converged, 0: go on, -1: failed
    __device__ int test(double h, int n) {
        constexpr double lo = sizeof(T) == 8 ? 1e-24 : 1e-11, hi = sizeof(T) == 8 ? 1e-12 : 1e-6;
        if (extra > 0) {
            --extra;
            return 0;
        }
        if (!(h < INFINITY)) return -1;
        if (h < lo * n || (h < hi * n && h > 0.25 * prev)) return 1;
        if (sizeof(T) == 4 && h < hi * n) extra = 1;  // this step and one more
        prev = h;
        return 0;
    }
};

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
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

// C = A B of matrices in shared memory (rows of pitch P, zero past N), NB x NB
// outputs a thread of 16 x 16 (rows ty + 16 i, columns NB tx + j); f(m, n, value)
// for every output.
template <typename T, int NB, int P, class F>
__device__ __forceinline__ void one_product(int N, const T* A, const T* B, F f) {
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    constexpr int KV = sizeof(T) == 4 ? 4 : 1;
    T acc[NB][NB];
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) acc[i][j] = T(0);
    for (int k = 0; k < N; k += KV) {
        T a[NB][KV], b[KV][NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) load_row<T, KV>(A + (ty + 16 * i) * P + k, a[i]);
#pragma unroll
        for (int q = 0; q < KV; ++q) load_row<T, NB>(B + (k + q) * P + NB * tx, b[q]);
#pragma unroll
        for (int q = 0; q < KV; ++q)
#pragma unroll
            for (int i = 0; i < NB; ++i)
#pragma unroll
                for (int j = 0; j < NB; ++j) acc[i][j] = fma(a[i][q], b[q][j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int m = ty + 16 * i, n = NB * tx + j;
            if (m < N && n < N) f(m, n, acc[i][j]);
        }
}

template <typename T, int NB>
__global__ void __launch_bounds__(kNsThreads) ns_one_kernel(int N, const double* __restrict__ A, double* __restrict__ X,
                                                            int* status) {
    constexpr int R = 16 * NB, P = R + (sizeof(T) == 4 ? 4 : 1);
    extern __shared__ double ns_smem[];
    __shared__ double sh[kNsThreads / 32];
    T* Y = reinterpret_cast<T*>(ns_smem);
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
        double h = 0.0;
        one_product<T, NB, P>(N, Z, Y, [&](int m, int n, T v) {
            const T d = m == n ? T(1) : T(0);
            const double x = (double)(d - v);
            h += x * x;
            W[m * P + n] = T(0.5) * (T(2) * d + (d - v));  // (3 delta - v) / 2
        });
        h = block_sum(h, sh);
        const int st = stop.test(h, N);
        if (st != 0) {
            ok = st > 0;
            break;
        }
        __syncthreads();
        one_product<T, NB, P>(N, Y, W, [&](int m, int n, T v) { Y2[m * P + n] = v; });
        one_product<T, NB, P>(N, W, Z, [&](int m, int n, T v) { Z2[m * P + n] = v; });
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
    double* part;              // one a CTA
    unsigned* bar;             // 4, zero at launch
    unsigned long long* norm;  // zero at launch
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
    __shared__ double sh[kNsThreads / 32];
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
    if (!grid_barrier(a.bar, gen, &abort_sh)) return;
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
    if (!grid_barrier(a.bar, gen, &abort_sh)) return;
    T *Y = a.Y, *Z = a.Z, *Y2 = a.Y2, *Z2 = a.Z2;
    auto put = [&](T* M, int m, int n, T v) { __stcg(M + (size_t)m * ld + n, v); };
    // sum over the CTAs in a fixed order: every CTA decides alike
    auto total = [&]() {
        double s = 0.0;
        if (warp == 0) {
            for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(a.part + b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) sh[0] = s;
        }
        __syncthreads();
        s = sh[0];
        __syncthreads();
        return s;
    };
    Stop<T> stop;
    bool ok = false;
    for (int it = 0; it < kNsMaxIt; ++it) {
        if (stop.done()) {
            ok = true;
            break;
        }
        if (it > 0) {
            double h = 0.0;
            for (int t = blockIdx.x; t < tiles; t += gridDim.x)
                grid_product<T>(N, ld, Z, Y, t / nt, t % nt, smem, [&](int m, int n, T v) {
                    const T d = m == n ? T(1) : T(0);
                    const double x = (double)(d - v);
                    h += x * x;
                    put(a.W, m, n, T(0.5) * (T(2) * d + (d - v)));
                });
            h = block_sum(h, sh);
            if (tid == 0) __stcg(a.part + blockIdx.x, h);
            if (!grid_barrier(a.bar, gen, &abort_sh)) return;
            const int st = stop.test(total(), N);
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
        if (!grid_barrier(a.bar, gen, &abort_sh)) return;
        T* t = Y;
        Y = Y2;
        Y2 = t;
        t = Z;
        Z = Z2;
        Z2 = t;
    }
    // ||(A/c)^{-1/2}||_F^2 >= lambda_max / lambda_min: reject ill-conditioned A
    double f = 0.0;
    const double s = 1.0 / sqrt(c);
    for (size_t e = me; e < (size_t)N * N; e += all) {
        const double z = 0.5 * ((double)__ldcg(Z + (e / N) * ld + e % N) + (double)__ldcg(Z + (e % N) * ld + e / N));
        f += z * z;
        if (ok) a.X[e] = s * z;
    }
    f = block_sum(f, sh);
    if (tid == 0) __stcg(a.part + blockIdx.x, f);
    if (!grid_barrier(a.bar, gen, &abort_sh)) return;
    f = total();
    if (me == 0) *a.status = ok && f < 1e12 ? 1 : 0;
}

template <typename T, int NB>
cudaError_t ns_one(int N, const double* A, double* X, int* d_status, cudaStream_t s) {
    constexpr int R = 16 * NB, P = R + (sizeof(T) == 4 ? 4 : 1);
    constexpr size_t sm = 5 * sizeof(T) * R * P;
    const void* fn = (const void*)ns_one_kernel<T, NB>;
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e) return e;
    }
    ns_one_kernel<T, NB><<<1, kNsThreads, sm, s>>>(N, A, X, d_status);
    return cudaGetLastError();
}

// X = A^{-1/2}; work: five N x ld matrices of T, then the control words.
template <typename T>
cudaError_t inv_sqrt(int N, const double* A, double* X, double* work, int* ok, cudaStream_t s, int* launches) {
    *ok = 0;
    const int ld = sizeof(T) == 4 ? (N + 3) / 4 * 4 : N;
    const size_t mat = ((size_t)N * ld * sizeof(T) + 15) / 16 * 16;
    unsigned char* w = reinterpret_cast<unsigned char*>(((uintptr_t)work + 15) & ~(uintptr_t)15);
    unsigned char* ctl = w + 5 * mat;
    int* d_status = reinterpret_cast<int*>(ctl);
    cudaError_t e;
    int h = 0;
    const bool one = sizeof(T) == 4 ? N <= 64 : N <= 16;
    if (one) {
        if (sizeof(T) == 8 || N <= 16) e = ns_one<T, 1>(N, A, X, d_status, s);
        else if (N <= 32) e = ns_one<float, 2>(N, A, X, d_status, s);
        else if (N <= 48) e = ns_one<float, 3>(N, A, X, d_status, s);
        else e = ns_one<float, 4>(N, A, X, d_status, s);
        if (e) return e;
    } else {
        if ((e = cudaMemsetAsync(ctl, 0xff, sizeof(int), s))) return e;        // status -1
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
        a.part = reinterpret_cast<double*>(ctl + 64);
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
    if ((e = cudaMemcpyAsync(&h, d_status, sizeof(int), cudaMemcpyDeviceToHost, s))) return e;
    if ((e = cudaStreamSynchronize(s))) return e;
    if (h < 0) return cudaErrorLaunchTimeout;  // a barrier wait ran out
    *ok = h == 1;
    return cudaSuccess;
}

}  // namespace

cudaError_t inv_sqrt_spd(int N, const double* A, double* X, double* work, int* ok, cudaStream_t s, int* launches) {
    return inv_sqrt<double>(N, A, X, work, ok, s, launches);
}
cudaError_t inv_sqrt_spd_mixed(int N, const double* A, double* X, double* work, int* ok, cudaStream_t s, int* launches) {
    return inv_sqrt<float>(N, A, X, work, ok, s, launches);
}

}  // namespace lace
