// The lane passes (pairconv_lanes.cuh) for grids whose sizes are known only
// at run time: orthorhombic boxes, and cubes without kernels of their own.
// The radices are dispatched per stage to the same butterflies; sizes and
// strides are kernel arguments.
#pragma once

#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

// First entry of axis n in the concatenated tables, and their length.
__host__ __device__ constexpr int box_offset(int n) {
    int o = 0;
    for (int k = 4; k < n; ++k)
        if (radices(k).big) o += k;
    return o;
}
constexpr int kBoxTw = box_offset(kMaxN + 1), kBoxLane = box_offset(kMaxN / 2 + 1);
struct BoxTables {
    float tw[kBoxTw][4];
    float lane[kBoxLane][2];
};
constexpr BoxTables make_box_tables() {
    BoxTables b{};
    int o = 0;
    for (int n = 4; n <= kMaxN; ++n) {
        const Radices r = radices(n);
        if (!r.big) continue;
        for (int e = 0; e < n; ++e) {
            const int m = (e / r.small) * (e % r.small);
            b.tw[o + e][0] = b.tw[o + e][1] = (float)ct_cos2pi(m, n);
            b.tw[o + e][2] = b.tw[o + e][3] = (float)-ct_sin2pi(m, n);
            if (n <= kMaxN / 2) {
                const int k = slot_k(e, r.big, r.small);
                b.lane[o + e][0] = (float)ct_cos2pi(k, 2 * n);
                b.lane[o + e][1] = (float)-ct_sin2pi(k, 2 * n);
            }
        }
        o += n;
    }
    return b;
}
__constant__ const BoxTables c_box = make_box_tables();

// Geometry of a plane of NY rows of NZ points.  Divisions by a size d
// multiply by ceil(2^22 / d): exact for items below 2^15 and d <= 128.
struct Box {
    int NY, NZ, H, PR, R1Z, R2Z, R1Y, R2Y;
    unsigned mny, mh, mhh;
    int oz, oy;
    bool kVec4;
    static __device__ __forceinline__ void split(int item, int d, unsigned m, int& q, int& r) {
        q = (int)(((unsigned)item * m) >> 22);
        r = item - q * d;
    }
    __device__ __forceinline__ void by_ny(int item, int& q, int& r) const { split(item, NY, mny, q, r); }
    __device__ __forceinline__ void by_h(int item, int& q, int& r) const { split(item, H, mh, q, r); }
    __device__ __forceinline__ void by_hh(int item, int& q, int& r) const { split(item, H / 2, mhh, q, r); }
    __device__ __forceinline__ Tw4 twz() const { return c_box.tw + oz; }
    __device__ __forceinline__ Tw4 twy() const { return c_box.tw + oy; }
    __device__ __forceinline__ Tw2 lane() const { return c_box.lane + oz; }
};
inline Box make_box(int ny, int nz) {
    Box b{};
    b.NY = ny;
    b.NZ = nz;
    b.H = nz / 2;
    b.PR = b.H | 1;
    const Radices z = radices(b.H), y = radices(ny);
    b.R1Z = z.big;
    b.R2Z = z.small;
    b.R1Y = y.small;
    b.R2Y = y.big;
    auto magic = [](int d) { return d > 0 ? (unsigned)(((1u << 22) + d - 1) / d) : 0u; };
    b.mny = magic(ny);
    b.mh = magic(b.H);
    b.mhh = magic(b.H / 2);
    b.oz = box_offset(b.H);
    b.oy = box_offset(ny);
    b.kVec4 = nz % 4 == 0;
    return b;
}

#define LN_SMALL(R_, F)                                                                              \
    switch (R_) {                                                                                    \
        case 2: F(2); break; case 3: F(3); break; case 4: F(4); break; case 5: F(5); break;          \
        case 6: F(6); break; case 8: F(8); break; case 9: F(9); break; default: F(10); break;        \
    }
#define LN_BIG(R_, F)                                                                                \
    switch (R_) {                                                                                    \
        case 2: F(2); break; case 3: F(3); break; case 4: F(4); break; case 5: F(5); break;          \
        case 6: F(6); break; case 8: F(8); break; case 9: F(9); break; case 10: F(10); break;        \
        case 12: F(12); break; case 15: F(15); break; default: F(16); break;                         \
    }

// Up to 768 threads of 80 registers: the warps of one CTA, or of several
// smaller ones, fill an SM's register file.  Against the kernels of a cube
// (us a grid, passes A and C): 72^3 1.29 and 1.96 against 1.18 and 1.77, 96^3
// 2.96 and 4.51 against 2.95 and 4.12, 48^3 0.37 and 0.61 against 0.35 and 0.53.
constexpr int kBoxRegs = 80, kBoxMaxThreads = 768;
template <int REGS>
__global__ void __launch_bounds__(kBoxMaxThreads) __maxnreg__(REGS) box_a(ConvArgs<float> P, int g0, Box g) {
    extern __shared__ P16 smem[];
    const int x = blockIdx.y, tid = threadIdx.x, nt = blockDim.x, n1 = gridDim.y;
    const GridView V = grid_view(P, g0, blockIdx.x, n1);
    load_rho(g, P, V, x, smem, tid, nt);
    prefetch_orbitals(g, P, g0, n1);
    __syncthreads();
#define LN_F(R) z_strided<R, -1>(g, smem, tid, nt)
    LN_BIG(g.R1Z, LN_F)
#undef LN_F
    __syncthreads();
#define LN_F(R) z_blocks<R, -1>(g, smem, tid, nt)
    LN_SMALL(g.R2Z, LN_F)
#undef LN_F
    __syncthreads();
#define LN_F(R) y_strided<R, -1>(g, smem, tid, nt)
    LN_SMALL(g.R1Y, LN_F)
#undef LN_F
    __syncthreads();
    P16* out = V.scr + (size_t)x * g.NY * g.H;
#define LN_F(R) y_blocks<R, -1>(g, smem, out, tid, nt)
    LN_BIG(g.R2Y, LN_F)
#undef LN_F
}

template <int REGS>
__global__ void __launch_bounds__(kBoxMaxThreads) __maxnreg__(REGS) box_c(ConvArgs<float> P, int g0, Box g) {
    extern __shared__ P16 smem[];
    __shared__ double red[64];
    const int x = blockIdx.y, tid = threadIdx.x, nt = blockDim.x, n1 = gridDim.y;
    const GridView V = grid_view(P, g0, blockIdx.x, n1);
    const size_t m = (size_t)g.NY * g.H;
    {
        int xa = 0, ga = 0;
        if (tid == 32 && ahead_cta(P.pf_ahead, ga, xa)) prefetch_l2(grid_view(P, g0, ga, n1).scr + xa * m, (unsigned)(m * 16));
    }
    P16* in = V.scr + (size_t)x * m;
#define LN_F(R) y_blocks<R, +1>(g, smem, in, tid, nt)
    LN_BIG(g.R2Y, LN_F)
#undef LN_F
    prefetch_epilogue(g, P, V, x, tid);
    __syncthreads();
#define LN_F(R) y_strided<R, +1>(g, smem, tid, nt)
    LN_SMALL(g.R1Y, LN_F)
#undef LN_F
    __syncthreads();
#define LN_F(R) z_blocks<R, +1>(g, smem, tid, nt)
    LN_SMALL(g.R2Z, LN_F)
#undef LN_F
    __syncthreads();
#define LN_F(R) z_strided<R, +1>(g, smem, tid, nt)
    LN_BIG(g.R1Z, LN_F)
#undef LN_F
    __syncthreads();
    store_w(g, P, V, x, smem, red, tid, nt);
}

}  // namespace ln
}  // namespace lace
