// FP32 passes of the pair convolutions (Eq. 2 evaluated with FFTs, Sec. 2;
// truncated by Eq. 5) with two lines of a grid in the lanes of every packed
// FP32 instruction (dft_lanes.cuh).  Any grid whose z size is even and whose
// axes factor into two radices up to 16; the bodies are templates on a
// geometry whose sizes are compile-time constants (Cube) or run-time values
// (Box).
//
// Layout.  A pair of points is 16 bytes: (re, re, im, im).  In real space the
// lanes are z = 2c and 2c + 1, the order in which orbitals lie in memory; the
// z transform runs length H = n3/2 on both lanes at once (the even and the odd
// points) and ends with the radix-2 step across the lanes, after which the
// lanes are kz = c and c + H.  The y and x transforms take a pair of columns
// (c, c + H) as it is.
//
// In place.  An axis of N = R1 R2 runs as R1-point DFTs over elements
// i + t R2 (i < R2), products with w_N^{i k1}, and R2-point DFTs over the
// blocks k1 R2 + i: every butterfly writes the slots that it read, so one
// plane buffer serves all stages, a stage ends in one barrier, and the result
// k = k1 + R1 k2 stands in slot k1 R2 + k2.  Reciprocal space stays in that
// order on all three axes (the table of K is laid out to match), and the
// inverse transform runs the stages backwards to natural order.  One buffer
// instead of two lets twice the CTAs share an SM (three at 72^3 instead of
// two, two at 96^3 instead of one, and 120^3 and 128^3 fit at all).
//
// The table holds -K(G)/Ng, so pass C adds psi v to W without a sign change.
//
// Bank conflicts: z stages run with consecutive threads on consecutive rows
// (odd row pitch in 16-byte units), y and x stages with consecutive threads
// on consecutive columns, so the eight 16-byte accesses of each
// quarter-warp phase fall on distinct bank groups, and the stage's twiddle
// factors are the same for (nearly) a whole warp: broadcast reads.
#pragma once

#include <atomic>

#include "dft_lanes.cuh"
#include "lace_internal.cuh"

namespace lace {
namespace ln {

using lanes::D;
using lanes::V2;
using lanes::ld2;
using lanes::st2;
using P16 = ulonglong2;  // one pair of points

// Packed instructions a point of an R-point butterfly, in hundredths.
__host__ __device__ constexpr int radix_cost(int r) {
    switch (r) {
        case 1: return 0;
        case 2: return 100;
        case 3: return 267;
        case 4: return 200;
        case 5: return 520;
        case 6: return 367;
        case 8: return 375;
        case 9: return 710;
        case 10: return 620;
        case 12: return 467;
        case 15: return 880;
        case 16: return 680;
        default: return 1 << 20;
    }
}
struct Radices {
    int big, small;
};
// The two radices of n with the fewest instructions; {0, 0}: none.
__host__ __device__ constexpr Radices radices(int n) {
    Radices best{0, 0};
    int cost = 1 << 20;
    for (int a = 2; a <= 16; ++a) {
        if (n % a) continue;
        const int b = n / a;
        if (b > a || b < 2) continue;
        const int c = radix_cost(a) + radix_cost(b);
        if (c < cost) {
            cost = c;
            best = Radices{a, b};
        }
    }
    return best;
}
// Slot s of an axis of r1 * r2 holds frequency slot_k(s).
__host__ __device__ constexpr int slot_k(int s, int r1, int r2) { return s / r2 + r1 * (s % r2); }

// Twiddle factors of an axis of n = big * small points, applied by the stage
// of the smaller radix: entry [i < big][t < small] = w_n^{i t} (forward sign)
// as (c, c, s, s), in constant memory: the factor is the same for most of a
// warp, and reading it through the constant cache keeps it off the
// shared-memory pipe that bounds the passes (a broadcast 16-byte shared read
// costs as much of it as the data).
template <int N> struct TwTable {
    float v[N][4];
};
template <int N> constexpr TwTable<N> make_tw() {
    TwTable<N> t{};
    constexpr int r = radices(N).small;
    for (int e = 0; e < N; ++e) {
        const int m = (e / r) * (e % r);
        t.v[e][0] = t.v[e][1] = (float)ct_cos2pi(m, N);
        t.v[e][2] = t.v[e][3] = (float)-ct_sin2pi(m, N);
    }
    return t;
}
template <int N> __constant__ const TwTable<N> c_tw = make_tw<N>();
// The factors of the step across the lanes in slot order: w_{2 H}^{k(s)}.
template <int H> struct LaneTable {
    float v[H][2];
};
template <int H> constexpr LaneTable<H> make_lane() {
    LaneTable<H> t{};
    for (int s = 0; s < H; ++s) {
        const int k = slot_k(s, radices(H).big, radices(H).small);
        t.v[s][0] = (float)ct_cos2pi(k, 2 * H);
        t.v[s][1] = (float)-ct_sin2pi(k, 2 * H);
    }
    return t;
}
template <int H> __constant__ const LaneTable<H> c_lane = make_lane<H>();
using Tw4 = const float (*)[4];
using Tw2 = const float (*)[2];

// Compile-time geometry of a plane of NY rows of NZ points.
template <int NY_, int NZ_> struct Plane {
    static constexpr int NY = NY_, NZ = NZ_, H = NZ_ / 2, PR = H | 1;
    static constexpr int R1Z = radices(H).big, R2Z = radices(H).small;
    static constexpr int R1Y = radices(NY_).small, R2Y = radices(NY_).big;
    static constexpr bool kVec4 = NZ_ % 4 == 0;
    static __device__ __forceinline__ void by_ny(int item, int& q, int& r) { q = item / NY; r = item % NY; }
    static __device__ __forceinline__ void by_h(int item, int& q, int& r) { q = item / H; r = item % H; }
    static __device__ __forceinline__ void by_hh(int item, int& q, int& r) { q = item / (H / 2); r = item % (H / 2); }
    static __device__ __forceinline__ Tw4 twz() { return c_tw<H>.v; }
    static __device__ __forceinline__ Tw4 twy() { return c_tw<NY>.v; }
    static __device__ __forceinline__ Tw2 lane() { return c_lane<H>.v; }
};
// 16-byte units of the plane buffer and the tables after it
__host__ __device__ constexpr size_t plane_smem(int ny, int nz) {
    const size_t h = nz / 2;
    return 16 * (size_t)ny * (h | 1);
}
__host__ __device__ constexpr size_t slab_smem(int nx, int lb) { return 16 * (size_t)nx * lb; }

__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// A plane of n floats: the 16-byte units that lie inside it (planes of an odd
// number of point pairs start between two units).
__device__ __forceinline__ void prefetch_plane(const float* p, size_t n) {
    const uintptr_t a = ((uintptr_t)p + 15) & ~(uintptr_t)15, e = (uintptr_t)(p + n) & ~(uintptr_t)15;
    prefetch_l2(reinterpret_cast<const void*>(a), (unsigned)(e - a));
}
__device__ __forceinline__ bool ahead_cta(int pf_ahead, int& fast, int& slow) {
    if (pf_ahead <= 0) return false;
    const long lin = (long)blockIdx.y * gridDim.x + blockIdx.x + pf_ahead;
    if (lin >= (long)gridDim.x * gridDim.y) return false;
    fast = (int)(lin % gridDim.x);
    slow = (int)(lin / gridDim.x);
    return true;
}

// The buffers of grid g of a launch (its own system's in a merged launch).
struct GridView {
    const float* psi;
    float* W;
    const float* ktab;
    P16* scr;
    double* ep;
    PairGrid d;
    int n_occ;
    double dv;
};
__device__ __forceinline__ GridView grid_view(const ConvArgs<float>& P, int g0, int g, int n1) {
    GridView v;
    if (P.refs) {
        const GridRef r = P.refs[g0 + g];
        const MergedSys<float>& m = P.msys[r.sys];
        v.psi = m.psi;
        v.W = m.W;
        v.ktab = m.klanes;
        v.d = m.grids[r.g];
        v.scr = reinterpret_cast<P16*>(m.scratch + (size_t)(r.g - m.g0) * P.ng);
        v.ep = m.epart + (size_t)(r.g - m.g0) * n1 * 2;
        v.n_occ = m.n_occ;
        v.dv = m.dv;
    } else {
        v.psi = P.psi;
        v.W = P.W;
        v.ktab = P.klanes;
        v.d = P.grids[g0 + g];
        v.scr = reinterpret_cast<P16*>(P.scratch + (size_t)g * P.ng);
        v.ep = P.epart + (size_t)g * n1 * 2;
        v.n_occ = P.n_occ;
        v.dv = P.dv;
    }
    return v;
}

// Products with the R factors at tw (one 16-byte entry (c, c, s, s) each,
// the first trivial).
template <int R, int DIR> __device__ __forceinline__ void twiddles(V2* v, Tw4 tw) {
#pragma unroll
    for (int t = 1; t < R; ++t) v[t] = lanes::cmulw<DIR>(v[t], mk2(tw[t][0], tw[t][1]), mk2(tw[t][2], tw[t][3]));
}

// The radix-2 step across the lanes.  Forward: lanes (even, odd) spectra ->
// (X[k], X[k + H]) = (E + w O, E - w O), w = (c, s).
__device__ __forceinline__ V2 lanes_join(V2 v, float2 w) {
    float er, od, ei, oi;
    unpk2(v.re, er, od);
    unpk2(v.im, ei, oi);
    const float tr = od * w.x - oi * w.y, ti = od * w.y + oi * w.x;
    return V2{mk2(er + tr, er - tr), mk2(ei + ti, ei - ti)};
}
// Inverse: (X[k], X[k + H]) -> spectra of the even and the odd points.
__device__ __forceinline__ V2 lanes_split(V2 v, float2 w) {
    float r0, r1, i0, i1;
    unpk2(v.re, r0, r1);
    unpk2(v.im, i0, i1);
    const float dr = r0 - r1, di = i0 - i1;
    return V2{mk2(r0 + r1, dr * w.x + di * w.y), mk2(i0 + i1, di * w.x - dr * w.y)};
}

// The stages of a plane.  z: R1 is the larger radix (strided stage), y: the
// smaller; the twiddles go with the smaller one.  Forward: strided, then
// blocks; inverse: blocks, then strided.
template <int R, int DIR, class G> __device__ __forceinline__ void z_strided(const G& g, P16* b, int tid, int nt) {
    for (int item = tid; item < g.NY * g.R2Z; item += nt) {
        int i, y;
        g.by_ny(item, i, y);
        P16* p = b + y * g.PR + i;
        V2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = ld2(p + t * g.R2Z);
        D<R, DIR>::run(v);
#pragma unroll
        for (int t = 0; t < R; ++t) st2(p + t * g.R2Z, v[t]);
    }
}
template <int R, int DIR, class G> __device__ __forceinline__ void z_blocks(const G& g, P16* b, int tid, int nt) {
    for (int item = tid; item < g.NY * g.R1Z; item += nt) {
        int k1, y;
        g.by_ny(item, k1, y);
        P16* p = b + y * g.PR + k1 * R;
        const Tw2 w = g.lane() + k1 * R;
        V2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            v[t] = ld2(p + t);
            if constexpr (DIR > 0) v[t] = lanes_split(v[t], make_float2(w[t][0], w[t][1]));
        }
        if constexpr (DIR < 0) twiddles<R, DIR>(v, g.twz() + k1 * R);
        D<R, DIR>::run(v);
        if constexpr (DIR > 0) twiddles<R, DIR>(v, g.twz() + k1 * R);
#pragma unroll
        for (int t = 0; t < R; ++t) {
            if constexpr (DIR < 0) v[t] = lanes_join(v[t], make_float2(w[t][0], w[t][1]));
            st2(p + t, v[t]);
        }
    }
}
template <int R, int DIR, class G> __device__ __forceinline__ void y_strided(const G& g, P16* b, int tid, int nt) {
    for (int item = tid; item < g.H * g.R2Y; item += nt) {
        int i, c;
        g.by_h(item, i, c);
        const int step = g.R2Y * g.PR;
        P16* p = b + i * g.PR + c;
        V2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = ld2(p + t * step);
        if constexpr (DIR > 0) twiddles<R, DIR>(v, g.twy() + i * R);
        D<R, DIR>::run(v);
        if constexpr (DIR < 0) twiddles<R, DIR>(v, g.twy() + i * R);
#pragma unroll
        for (int t = 0; t < R; ++t) st2(p + t * step, v[t]);
    }
}
// forward: shared memory -> global rows; inverse: global rows -> shared memory
template <int R, int DIR, class G> __device__ __forceinline__ void y_blocks(const G& g, P16* b, P16* glob, int tid, int nt) {
    for (int item = tid; item < g.H * g.R1Y; item += nt) {
        int k1, c;
        g.by_h(item, k1, c);
        P16* p = b + k1 * R * g.PR + c;
        P16* q = glob + k1 * R * g.H + c;
        V2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = DIR < 0 ? ld2(p + t * g.PR) : ld2(q + t * g.H);
        D<R, DIR>::run(v);
#pragma unroll
        for (int t = 0; t < R; ++t) {
            if constexpr (DIR < 0) st2(q + t * g.H, v[t]);
            else st2(p + t * g.PR, v[t]);
        }
    }
}

// Pass A: rho of plane x of both pairs into the buffer, forward z and y.
template <class G> __device__ __forceinline__ void load_rho(const G& g, const ConvArgs<float>& P, const GridView& V, int x, P16* buf, int tid, int nt) {
    const PairGrid d = V.d;
    const size_t off = (size_t)x * g.NY * g.NZ;
    const bool two = d.j2 >= 0;
    const float* a1 = V.psi + (size_t)d.i1 * P.ng + off;
    const float* c1 = V.psi + (size_t)d.j1 * P.ng + off;
    const float* a2 = V.psi + (size_t)(two ? d.i2 : d.i1) * P.ng + off;
    const float* c2 = V.psi + (size_t)(two ? d.j2 : d.j1) * P.ng + off;
    const bool same_i = d.i1 == d.i2;
    if (g.kVec4) {  // two pairs a thread: 16-byte loads
        const P16 *A1 = reinterpret_cast<const P16*>(a1), *C1 = reinterpret_cast<const P16*>(c1);
        const P16 *A2 = reinterpret_cast<const P16*>(a2), *C2 = reinterpret_cast<const P16*>(c2);
        for (int e = tid; e < g.NY * (g.H / 2); e += nt) {
            const P16 x1 = __ldg(A1 + e), y1 = __ldg(C1 + e);
            P16 x2 = make_ulonglong2(0, 0), y2 = x2;
            if (two) {
                x2 = same_i ? x1 : __ldg(A2 + e);
                y2 = __ldg(C2 + e);
            }
            int y, q;
            g.by_hh(e, y, q);
            const V2 lo{f2{x1.x} * f2{y1.x}, f2{x2.x} * f2{y2.x}}, hi{f2{x1.y} * f2{y1.y}, f2{x2.y} * f2{y2.y}};
            // 32 bytes a thread: half of the threads write their upper pair
            // first, so each store's phases cover all bank groups
            P16* p = buf + y * g.PR + 2 * q;
            const bool sw = (q >> 2) & 1;
            st2(p + sw, sw ? hi : lo);
            st2(p + 1 - sw, sw ? lo : hi);
        }
        return;
    }
    using L = const unsigned long long*;
    for (int e = tid; e < g.NY * g.H; e += nt) {
        const f2 x1{__ldg((L)a1 + e)}, y1{__ldg((L)c1 + e)};
        f2 x2{0}, y2{0};
        if (two) {
            x2 = same_i ? x1 : f2{__ldg((L)a2 + e)};
            y2 = f2{__ldg((L)c2 + e)};
        }
        int y, c;
        g.by_h(e, y, c);
        st2(buf + y * g.PR + c, V2{x1 * y1, x2 * y2});
    }
}

// Compensated sum of both lanes.
__device__ __forceinline__ void kahan2(f2& s, f2& c, f2 v) {
    const f2 y = v - c;
    const f2 t = s + y;
    c = (t - s) - y;
    s = t;
}
__device__ __forceinline__ void red4(float* p, f2 lo, f2 hi) {
    float4 v;
    unpk2(lo, v.x, v.y);
    unpk2(hi, v.z, v.w);
    atomicAdd(reinterpret_cast<float4*>(p), v);
}
__device__ __forceinline__ void red2(float* p, f2 a) {
    float2 v;
    unpk2(a, v.x, v.y);
    atomicAdd(reinterpret_cast<float2*>(p), v);
}

// Pass C after the transforms: buf holds -v (lanes z = 2c, 2c + 1; real part
// of pair a, imaginary part of pair b): W_j += w_i (-v) and, for an occupied
// j != i, W_i += psi_j (-v); the pair energies dV sum rho v to ep.
// red: 64 doubles of shared memory.
template <class G> __device__ __forceinline__ void store_w(const G& g, const ConvArgs<float>& P, const GridView& V, int x, const P16* buf, double* red, int tid, int nt) {
    const PairGrid d = V.d;
    const size_t off = (size_t)x * g.NY * g.NZ;
    const bool two = d.j2 >= 0;
    const bool a_occ = d.j1 < V.n_occ, a_sym = a_occ && d.j1 != d.i1;
    const bool b_occ = two && d.j2 < V.n_occ, b_sym = b_occ && d.j2 != d.i2;
    const size_t oi1 = (size_t)d.i1 * P.ng + off, oj1 = (size_t)d.j1 * P.ng + off;
    const size_t oi2 = (size_t)(two ? d.i2 : d.i1) * P.ng + off, oj2 = (size_t)(two ? d.j2 : d.j1) * P.ng + off;
    const bool same_i = d.i1 == d.i2;
    const bool merge_i = two && a_sym && b_sym && same_i;  // both add to the same W_i: one reduction
    f2 sa = bc2(0.f), ca = sa, sb = sa, cb = sa;
    if (g.kVec4) {
        for (int e = tid; e < g.NY * (g.H / 2); e += nt) {
            int y, q;
            g.by_hh(e, y, q);
            const P16* p = buf + y * g.PR + 2 * q;
            const bool sw = (q >> 2) & 1;
            const V2 p0 = ld2(p + sw), p1 = ld2(p + 1 - sw);
            const V2 lo = sw ? p1 : p0, hi = sw ? p0 : p1;
            const P16 x1 = __ldg(reinterpret_cast<const P16*>(V.psi + oi1) + e);
            const P16 y1 = __ldg(reinterpret_cast<const P16*>(V.psi + oj1) + e);
            const f2 u0 = f2{x1.x} * lo.re, u1 = f2{x1.y} * hi.re;
            red4(V.W + oj1 + 4 * e, u0, u1);
            f2 w0 = f2{y1.x} * lo.re, w1 = f2{y1.y} * hi.re;
            if (a_sym && !merge_i) red4(V.W + oi1 + 4 * e, w0, w1);
            if (a_occ) kahan2(sa, ca, fma2(u1, f2{y1.y}, u0 * f2{y1.x}));
            if (two) {
                const P16 x2 = same_i ? x1 : __ldg(reinterpret_cast<const P16*>(V.psi + oi2) + e);
                const P16 y2 = __ldg(reinterpret_cast<const P16*>(V.psi + oj2) + e);
                const f2 t0 = f2{x2.x} * lo.im, t1 = f2{x2.y} * hi.im;
                red4(V.W + oj2 + 4 * e, t0, t1);
                if (merge_i) {
                    w0 = fma2(f2{y2.x}, lo.im, w0);
                    w1 = fma2(f2{y2.y}, hi.im, w1);
                    red4(V.W + oi1 + 4 * e, w0, w1);
                } else if (b_sym) {
                    red4(V.W + oi2 + 4 * e, f2{y2.x} * lo.im, f2{y2.y} * hi.im);
                }
                if (b_occ) kahan2(sb, cb, fma2(t1, f2{y2.y}, t0 * f2{y2.x}));
            }
        }
    } else {
        using L = const unsigned long long*;
        for (int e = tid; e < g.NY * g.H; e += nt) {
            int y, c;
            g.by_h(e, y, c);
            const V2 v = ld2(buf + y * g.PR + c);
            const f2 x1{__ldg((L)(V.psi + oi1) + e)}, y1{__ldg((L)(V.psi + oj1) + e)};
            const f2 u = x1 * v.re;
            red2(V.W + oj1 + 2 * e, u);
            f2 w = y1 * v.re;
            if (a_sym && !merge_i) red2(V.W + oi1 + 2 * e, w);
            if (a_occ) kahan2(sa, ca, u * y1);
            if (two) {
                const f2 x2 = same_i ? x1 : f2{__ldg((L)(V.psi + oi2) + e)};
                const f2 y2{__ldg((L)(V.psi + oj2) + e)};
                const f2 t = x2 * v.im;
                red2(V.W + oj2 + 2 * e, t);
                if (merge_i) red2(V.W + oi1 + 2 * e, fma2(y2, v.im, w));
                else if (b_sym) red2(V.W + oi2 + 2 * e, y2 * v.im);
                if (b_occ) kahan2(sb, cb, t * y2);
            }
        }
    }
    float s0, s1, c0, c1;
    unpk2(sa, s0, s1);
    unpk2(ca, c0, c1);
    float ea = (s0 - c0) + (s1 - c1);
    unpk2(sb, s0, s1);
    unpk2(cb, c0, c1);
    float eb = (s0 - c0) + (s1 - c1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ea += __shfl_xor_sync(0xffffffffu, ea, o);
        eb += __shfl_xor_sync(0xffffffffu, eb, o);
    }
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    if (lane == 0) {
        red[warp] = (double)ea;
        red[32 + warp] = (double)eb;
    }
    __syncthreads();
    if (warp == 0) {
        // the warp partials in FP64 across the lanes of one warp (a short
        // chain: FP64 issues slowly)
        double ta = lane < nw ? red[lane] : 0.0, tb = lane < nw ? red[32 + lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ta += __shfl_xor_sync(0xffffffffu, ta, o);
            tb += __shfl_xor_sync(0xffffffffu, tb, o);
        }
        if (lane == 0) {
            V.ep[(size_t)x * 2] = -ta * V.dv;
            V.ep[(size_t)x * 2 + 1] = -tb * V.dv;
        }
    }
}

// Pass B, columns j0 .. j0 + LB - 1 of the M columns of a plane: forward x
// (strided stage from global memory), then per block the R2-point DFT, the
// product with the table and the inverse R2-point DFT in registers, then
// the inverse strided stage back to global memory.  R1 >= R2.
template <int R1, int R2, int LB> struct Slab {
    static __device__ __forceinline__ void run(P16* __restrict__ base, int M, int j0, const unsigned long long* __restrict__ ktab, P16* b, int tid, int nt) {
        for (int item = tid; item < LB * R2; item += nt) {
            const int j = item % LB, i = item / LB;
            if (j0 + j < M) {
                P16* q = base + (size_t)i * M + j0 + j;
                V2 v[R1];
#pragma unroll
                for (int t = 0; t < R1; ++t) v[t] = ld2(q + (size_t)t * R2 * M);
                D<R1, -1>::run(v);
#pragma unroll
                for (int t = 0; t < R1; ++t) st2(b + (i + t * R2) * LB + j, v[t]);
            }
        }
        __syncthreads();
        for (int item = tid; item < LB * R1; item += nt) {
            const int j = item % LB, k1 = item / LB;
            if (j0 + j < M) {
                const unsigned long long* kp = ktab + (size_t)k1 * R2 * M + j0 + j;
                f2 k[R2];
#pragma unroll
                for (int t = 0; t < R2; ++t) k[t] = f2{__ldg(kp + (size_t)t * M)};
                P16* p = b + k1 * R2 * LB + j;
                V2 v[R2];
#pragma unroll
                for (int t = 0; t < R2; ++t) v[t] = ld2(p + t * LB);
                twiddles<R2, -1>(v, c_tw<R1 * R2>.v + k1 * R2);
                D<R2, -1>::run(v);
#pragma unroll
                for (int t = 0; t < R2; ++t) v[t] = V2{v[t].re * k[t], v[t].im * k[t]};
                D<R2, +1>::run(v);
                twiddles<R2, +1>(v, c_tw<R1 * R2>.v + k1 * R2);
#pragma unroll
                for (int t = 0; t < R2; ++t) st2(p + t * LB, v[t]);
            }
        }
        __syncthreads();
        for (int item = tid; item < LB * R2; item += nt) {
            const int j = item % LB, i = item / LB;
            if (j0 + j < M) {
                P16* q = base + (size_t)i * M + j0 + j;
                V2 v[R1];
#pragma unroll
                for (int t = 0; t < R1; ++t) v[t] = ld2(b + (i + t * R2) * LB + j);
                D<R1, +1>::run(v);
#pragma unroll
                for (int t = 0; t < R1; ++t) st2(q + (size_t)t * R2 * M, v[t]);
            }
        }
    }
};

// ------------------------------------------------------------------ kernels
template <class G> __device__ __forceinline__ void prefetch_orbitals(const G& g, const ConvArgs<float>& P, int g0, int n1) {
    int xa = 0, ga = 0;
    if (threadIdx.x < 4 && ahead_cta(P.pf_ahead, ga, xa)) {
        const GridView A = grid_view(P, g0, ga, n1);
        const int o = threadIdx.x == 0 ? A.d.i1 : threadIdx.x == 1 ? A.d.j1 : threadIdx.x == 2 ? A.d.i2 : A.d.j2;
        const size_t np = (size_t)g.NY * g.NZ;
        if (o >= 0) prefetch_plane(A.psi + (size_t)o * P.ng + xa * np, np);
    }
}

// Pass C's orbital and W planes, fetched into L2 while its stages run.
template <class G> __device__ __forceinline__ void prefetch_epilogue(const G& g, const ConvArgs<float>& P, const GridView& V, int x, int tid) {
    if (P.pf_ahead > 0 && tid < 8) {
        const int q = tid & 3;
        const int o = q == 0 ? V.d.i1 : q == 1 ? V.d.j1 : q == 2 ? V.d.i2 : V.d.j2;
        const size_t np = (size_t)g.NY * g.NZ;
        if (o >= 0) prefetch_plane((tid < 4 ? V.psi : V.W) + (size_t)o * P.ng + x * np, np);
    }
}

template <int N, int NT, int REGS>
__global__ void __launch_bounds__(NT) __maxnreg__(REGS) cube_a(ConvArgs<float> P, int g0) {
    extern __shared__ P16 smem[];
    using G = Plane<N, N>;
    const G g;
    const int x = blockIdx.y, tid = threadIdx.x;  // plane-major: the CTAs in flight share plane x
    const GridView V = grid_view(P, g0, blockIdx.x, N);
    load_rho(g, P, V, x, smem, tid, NT);
    prefetch_orbitals(g, P, g0, N);
    __syncthreads();
    z_strided<G::R1Z, -1>(g, smem, tid, NT);
    __syncthreads();
    z_blocks<G::R2Z, -1>(g, smem, tid, NT);
    __syncthreads();
    y_strided<G::R1Y, -1>(g, smem, tid, NT);
    __syncthreads();
    y_blocks<G::R2Y, -1>(g, smem, V.scr + (size_t)x * N * G::H, tid, NT);
}

template <int N, int NT, int REGS>
__global__ void __launch_bounds__(NT) __maxnreg__(REGS) cube_c(ConvArgs<float> P, int g0) {
    extern __shared__ P16 smem[];
    __shared__ double red[64];
    using G = Plane<N, N>;
    const G g;
    const int x = blockIdx.y, tid = threadIdx.x;
    const GridView V = grid_view(P, g0, blockIdx.x, N);
    {
        int xa = 0, ga = 0;
        if (tid == 32 && ahead_cta(P.pf_ahead, ga, xa))
            prefetch_l2(grid_view(P, g0, ga, N).scr + (size_t)xa * N * G::H, N * G::H * 16);
    }
    y_blocks<G::R2Y, +1>(g, smem, V.scr + (size_t)x * N * G::H, tid, NT);
    prefetch_epilogue(g, P, V, x, tid);
    __syncthreads();
    y_strided<G::R1Y, +1>(g, smem, tid, NT);
    __syncthreads();
    z_blocks<G::R2Z, +1>(g, smem, tid, NT);
    __syncthreads();
    z_strided<G::R1Z, +1>(g, smem, tid, NT);
    __syncthreads();
    store_w(g, P, V, x, smem, red, tid, NT);
}

// Pass B: columns of the planes of a grid (M = n2 n3 / 2 of them), LB a CTA.
template <int N, int LB, int NT, int REGS>
__global__ void __launch_bounds__(NT) __maxnreg__(REGS) slab_b(ConvArgs<float> P, int g0, int M) {
    extern __shared__ P16 smem[];
    const GridView V = grid_view(P, g0, blockIdx.y, N);
    {
        int ja = 0, ga = 0;
        if (threadIdx.x < N && ahead_cta(P.pf_ahead, ja, ga)) {
            const int j = ja * LB, n = min(LB, M - j);
            prefetch_l2(grid_view(P, g0, ga, N).scr + (size_t)threadIdx.x * M + j, n * 16);
        }
    }
    constexpr Radices r = radices(N);
    Slab<r.big, r.small, LB>::run(V.scr, M, blockIdx.x * LB, reinterpret_cast<const unsigned long long*>(V.ktab), smem, threadIdx.x, NT);
}

// ------------------------------------------------------------------ launch shapes
// Registers a thread may use when m CTAs of nt threads share an SM: the
// register file is split over four sub-partitions of 16K registers, and every
// warp takes its registers from one of them.
constexpr int regs_at(int nt, int m) {
    const int per_part = (m * ((nt + 31) / 32) + 3) / 4;
    const int r = 16384 / (per_part * 32) / 8 * 8;
    return r > 128 ? 128 : r;
}
// CTAs of a plane pass that an SM's shared memory holds (227 KB, 1 KB
// reserved and 0.5 KB of static arrays each), at most 8.
constexpr int plane_ctas(int ny, int nz) {
    const int m = (int)((227u * 1024u) / (plane_smem(ny, nz) + 1536));
    return m > 8 ? 8 : m < 1 ? 1 : m;
}
// Threads of a plane pass.  Measured (pass A, us a grid, 128 / 160 / 192 / 224 /
// 256 / 384 threads): 72^3, five CTAs an SM, 1.29 / 1.20 / 1.18 / 1.21 / - / -;
// 96^3, three, - / 3.31 / 3.04 / 2.95 / 2.98 / 3.23; 48^3, 0.353 / 0.359 /
// 0.373 / 0.400; 120^3, one CTA: 768 threads 8.0, 640 8.4, 512 8.4.
constexpr int plane_threads(int ny, int nz) {
    switch (plane_ctas(ny, nz)) {
        case 1: return 768;
        case 2: return 384;
        case 3: return 256;
        case 4: return 224;
        case 5: return 192;
        case 6: return 160;
        default: return 128;
    }
}
// Columns of a pass-B CTA and its threads: one round of the outer stage
// (72^3: 32 columns, 192 threads 0.91 us a grid, at 16 columns 0.94, at 64
// 1.02; 96^3: 16 columns 2.42, 32 2.57).
constexpr int slab_cols(int n) { return radices(n).small <= 3 ? 64 : radices(n).small <= 6 ? 32 : 16; }
constexpr int slab_threads(int n) { return (slab_cols(n) * radices(n).small + 31) / 32 * 32; }
constexpr int slab_regs(int n) { return radices(n).big >= 15 ? 128 : radices(n).small >= 8 ? 96 : radices(n).small <= 4 ? 64 : 80; }

template <class K> void smem_opt_in(K k, size_t bytes) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}
// One bit per device: the attributes of a kernel family are set.
struct OncePerDevice {
    std::atomic<unsigned long long> done{0};
    template <class F> void run(F f) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 64 && (done.load() & (1ull << dev))) return;
        f();
        if (dev < 64) done.fetch_or(1ull << dev);
    }
};

// Threads of a plane pass whose launch does not fill the SMs (the exchange of a few
// pairs): a CTA's chain of stages is all that counts then, and a thread a butterfly
// of most stages makes it shortest, with two CTAs an SM up to 384 threads and one beyond.
// Pass A and C of one grid, us: 48^3 8.2 and 9.1 -> 6.1 and 7.3 (128 -> 288 threads), 64^3 9.2
// and 10.5 -> 6.7 and 7.7, 96^3 13.2 and 14.7 -> 9.8 and 11.4; of five grids at
// 48^3 (240 CTAs) 8.6 and 11.1 -> 6.7 and 9.0.  Launches that do not fit at once are
// slower with it (48^3, eight grids: 12.6 -> 14.4), and below 40 points an axis the
// stages have no more items than the narrow CTA has threads.
constexpr int wide_threads(int n) {
    const int t = n < 40 ? 0 : (n * n / 8 + 31) / 32 * 32;
    return t > 768 ? 768 : t;
}
constexpr int wide_ctas(int n) { return wide_threads(n) <= 384 ? 2 : 1; }

template <int N, int NT, int CTAS> void launch_cube_as(int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    constexpr int RG = regs_at(NT, CTAS);
    constexpr size_t sm = plane_smem(N, N);
    static OncePerDevice once;
    once.run([&] {
        smem_opt_in(cube_a<N, NT, RG>, sm);
        smem_opt_in(cube_c<N, NT, RG>, sm);
    });
    if (pass == 0) cube_a<N, NT, RG><<<dim3(nb, N), NT, sm, s>>>(P, g0);
    else cube_c<N, NT, RG><<<dim3(nb, N), NT, sm, s>>>(P, g0);
}
template <int N> bool launch_cube(int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    constexpr int NT = plane_threads(N, N), WIDE = wide_threads(N);
    if constexpr (WIDE > NT) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if ((long long)nb * N <= (long long)wide_ctas(N) * sms) {
            launch_cube_as<N, WIDE, wide_ctas(N)>(pass, nb, P, g0, s);
            return true;
        }
    }
    launch_cube_as<N, NT, plane_ctas(N, N)>(pass, nb, P, g0, s);
    return true;
}
template <int N> bool launch_slab(int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    constexpr int LB = slab_cols(N), NT = slab_threads(N), RG = slab_regs(N);
    constexpr size_t sm = slab_smem(N, LB);
    static OncePerDevice once;
    once.run([&] { smem_opt_in(slab_b<N, LB, NT, RG>, sm); });
    slab_b<N, LB, NT, RG><<<dim3((M + LB - 1) / LB, nb), NT, sm, s>>>(P, g0, M);
    return true;
}

// Passes A and C (pass 0, 2) of a cube with kernels of its own (false: none),
// of any box, and pass B along an x axis of n points.
bool cube_1(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool cube_2(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool cube_3(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool cube_4(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool slab_1(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool slab_2(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
bool slab_3(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);
void box_pass(int n1, int n2, int n3, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s);

}  // namespace ln
}  // namespace lace
