// In-register DFTs over two lines at once: a value holds the real parts of
// the two lines in one register pair and their imaginary parts in another,
// so every operation of a butterfly, the products by +-i included, is one
// packed FP32 instruction (add/sub/mul/fma .rn.f32x2) for both lines.
// Against one line with (re, im) in a pair (dft_packed.cuh), the additions
// a +- i b and the twiddle products are packed too, and one 16-byte access
// moves two complex values.
//
// Sizes with coprime factors (6 = 2 x 3, 10 = 2 x 5, 12 = 3 x 4, 15 = 3 x 5)
// use the prime-factor map, which has no inner twiddles: at 72 = 12 x 6 that
// is 8.3 packed instructions a point and transform against 10.9 for 8 x 9.
// Irrational constants are carried as hi + lo floats (f32x2.cuh).
#pragma once

#include "common.cuh"
#include "f32x2.cuh"

namespace lace {
namespace lanes {

struct V2 {
    f2 re, im;
};

__device__ __forceinline__ V2 ld2(const ulonglong2* p) {
    const ulonglong2 q = *p;
    return V2{f2{q.x}, f2{q.y}};
}
__device__ __forceinline__ void st2(ulonglong2* p, V2 v) { *p = make_ulonglong2(v.re.v, v.im.v); }

__device__ __forceinline__ V2 add(V2 a, V2 b) { return V2{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ V2 sub(V2 a, V2 b) { return V2{a.re - b.re, a.im - b.im}; }
// a + i S b
template <int S> __device__ __forceinline__ V2 addi(V2 a, V2 b) {
    if constexpr (S > 0) return V2{a.re - b.im, a.im + b.re};
    else return V2{a.re + b.im, a.im - b.re};
}
// c real constant
__device__ __forceinline__ V2 scale(V2 a, double c) { return V2{mulk2(a.re, c), mulk2(a.im, c)}; }

// v * (c + i s) for DIR < 0, v * (c - i s) for DIR > 0, the same for both
// lanes: cc = (c, c), ss = (s, s) (the table holds the forward factors).
template <int DIR> __device__ __forceinline__ V2 cmulw(V2 v, f2 cc, f2 ss) {
    float s0, s1;
    unpk2(ss, s0, s1);
    const f2 ns = mk2(-s0, -s1);
    if constexpr (DIR < 0) return V2{fma2(v.im, ns, v.re * cc), fma2(v.re, ss, v.im * cc)};
    else return V2{fma2(v.im, ss, v.re * cc), fma2(v.re, ns, v.im * cc)};
}

// exp(DIR 2 pi i M / N) * a, compile-time
template <int N, int M, int DIR> __device__ __forceinline__ V2 tw_ct(V2 a) {
    constexpr int m = ((M % N) + N) % N;
    if constexpr (m == 0) {
        return a;
    } else if constexpr (4 * m == N || 4 * m == 3 * N) {
        constexpr int S = (4 * m == N) ? DIR : -DIR;
        const f2 z = bc2(0.f);
        if constexpr (S > 0) return V2{z - a.im, a.re};
        else return V2{a.im, z - a.re};
    } else if constexpr ((8 * m) % N == 0) {
        constexpr int e8 = 8 * m / N;
        constexpr int cx = (e8 == 1 || e8 == 7) ? 1 : -1;
        constexpr int ss = DIR * ((e8 == 1 || e8 == 3) ? 1 : -1);
        constexpr double h = 0.707106781186547524400844362104849039;
        const f2 s = a.re + a.im, d = a.re - a.im;
        // (cx + i ss) h (re + i im) = h (cx re - ss im) + i h (ss re + cx im)
        if constexpr (cx * ss > 0) return V2{mulk2(d, cx * h), mulk2(s, cx * h)};
        else return V2{mulk2(s, cx * h), mulk2(d, ss * h)};
    } else {
        constexpr double c = ct_cos2pi(m, N);
        constexpr double s = DIR * ct_sin2pi(m, N);
        return V2{fmak2(a.re, c, mulk2(a.im, -s)), fmak2(a.re, s, mulk2(a.im, c))};
    }
}

template <int R, int DIR> struct D;

template <int DIR> struct D<2, DIR> {
    static __device__ __forceinline__ void run(V2* v) {
        const V2 a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    }
};
template <int DIR> struct D<3, DIR> {
    static __device__ __forceinline__ void run(V2* v) {
        constexpr double s3 = 0.866025403784438646763723170752936183;  // sin(2 pi/3)
        const V2 a = v[0], t1 = add(v[1], v[2]), e = scale(sub(v[1], v[2]), s3);
        const f2 mh = bc2(-0.5f);
        const V2 t2{fma2(t1.re, mh, a.re), fma2(t1.im, mh, a.im)};
        v[0] = add(a, t1);
        v[1] = addi<DIR>(t2, e);
        v[2] = addi<-DIR>(t2, e);
    }
};
template <int DIR> struct D<4, DIR> {
    static __device__ __forceinline__ void run(V2* v) {
        const V2 s0 = add(v[0], v[2]), d0 = sub(v[0], v[2]);
        const V2 s1 = add(v[1], v[3]), e = sub(v[1], v[3]);
        v[0] = add(s0, s1);
        v[2] = sub(s0, s1);
        v[1] = addi<DIR>(d0, e);
        v[3] = addi<-DIR>(d0, e);
    }
};
template <int DIR> struct D<5, DIR> {
    static __device__ __forceinline__ void run(V2* v) {
        constexpr double c1 = ct_cos2pi(1, 5), c2 = ct_cos2pi(2, 5);
        constexpr double s1 = ct_sin2pi(1, 5), s2 = ct_sin2pi(2, 5);
        const V2 a = v[0];
        const V2 p1 = add(v[1], v[4]), m1 = sub(v[1], v[4]);
        const V2 p2 = add(v[2], v[3]), m2 = sub(v[2], v[3]);
        const V2 r1{fmak2(p1.re, c1, fmak2(p2.re, c2, a.re)), fmak2(p1.im, c1, fmak2(p2.im, c2, a.im))};
        const V2 r2{fmak2(p1.re, c2, fmak2(p2.re, c1, a.re)), fmak2(p1.im, c2, fmak2(p2.im, c1, a.im))};
        const V2 q1{fmak2(m1.re, s1, mulk2(m2.re, s2)), fmak2(m1.im, s1, mulk2(m2.im, s2))};
        const V2 q2{fmak2(m1.re, s2, mulk2(m2.re, -s1)), fmak2(m1.im, s2, mulk2(m2.im, -s1))};
        v[0] = add(a, add(p1, p2));
        v[1] = addi<DIR>(r1, q1);
        v[4] = addi<-DIR>(r1, q1);
        v[2] = addi<DIR>(r2, q2);
        v[3] = addi<-DIR>(r2, q2);
    }
};
// R = A * B, coprime (prime-factor map, no twiddles): input index
// B a + A b, output index k = ka mod A, kb mod B.
__host__ __device__ constexpr int mod_inverse(int a, int m) {
    for (int x = 1; x < m; ++x)
        if (a * x % m == 1) return x;
    return 0;
}
template <int A, int B, int DIR> struct Pfa {
    static constexpr int EA = B * mod_inverse(B, A), EB = A * mod_inverse(A, B);
    static __device__ __forceinline__ void run(V2* v) {
        V2 y[A * B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            V2 u[A];
#pragma unroll
            for (int a = 0; a < A; ++a) u[a] = v[(B * a + A * b) % (A * B)];
            D<A, DIR>::run(u);
#pragma unroll
            for (int a = 0; a < A; ++a) y[b * A + a] = u[a];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            V2 u[B];
#pragma unroll
            for (int b = 0; b < B; ++b) u[b] = y[b * A + a];
            D<B, DIR>::run(u);
#pragma unroll
            for (int b = 0; b < B; ++b) v[(a * EA + b * EB) % (A * B)] = u[b];
        }
    }
};
template <int DIR> struct D<6, DIR> : Pfa<3, 2, DIR> {};
template <int DIR> struct D<10, DIR> : Pfa<5, 2, DIR> {};
template <int DIR> struct D<12, DIR> : Pfa<4, 3, DIR> {};
template <int DIR> struct D<15, DIR> : Pfa<5, 3, DIR> {};

// R = A * B, Cooley-Tukey in registers: t = B ta + tb, k = ka + A kb.
template <int A, int B, int TB, int KA, int DIR> struct CtTw {
    static __device__ __forceinline__ void run(const V2* u, V2* y) {
        y[TB * A + KA] = tw_ct<A * B, TB * KA, DIR>(u[KA]);
        if constexpr (KA + 1 < A) CtTw<A, B, TB, KA + 1, DIR>::run(u, y);
    }
};
template <int A, int B, int TB, int DIR> struct CtStep {
    static __device__ __forceinline__ void run(const V2* v, V2* y) {
        V2 u[A];
#pragma unroll
        for (int ta = 0; ta < A; ++ta) u[ta] = v[B * ta + TB];
        D<A, DIR>::run(u);
        CtTw<A, B, TB, 0, DIR>::run(u, y);
        if constexpr (TB + 1 < B) CtStep<A, B, TB + 1, DIR>::run(v, y);
    }
};
template <int A, int B, int DIR> struct Ct {
    static __device__ __forceinline__ void run(V2* v) {
        V2 y[A * B];
        CtStep<A, B, 0, DIR>::run(v, y);
#pragma unroll
        for (int ka = 0; ka < A; ++ka) {
            V2 u[B];
#pragma unroll
            for (int tb = 0; tb < B; ++tb) u[tb] = y[tb * A + ka];
            D<B, DIR>::run(u);
#pragma unroll
            for (int kb = 0; kb < B; ++kb) v[ka + A * kb] = u[kb];
        }
    }
};
template <int DIR> struct D<8, DIR> : Ct<4, 2, DIR> {};
template <int DIR> struct D<9, DIR> : Ct<3, 3, DIR> {};
template <int DIR> struct D<16, DIR> : Ct<4, 4, DIR> {};

}  // namespace lanes
}  // namespace lace
