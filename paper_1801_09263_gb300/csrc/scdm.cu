// SCDM localisation support (Sec. 2): pivoted QR (Businger-Golub, modified
// Gram-Schmidt with exact column norms at every step) on the grid subsample,
// and the gathers that feed it and the U = phi_C^T (phi_C phi_C^T)^{-1/2}
// rotation computed by the caller.
#include <algorithm>

#include "f32x2.cuh"
#include "grid_sync.cuh"
#include "lace_internal.cuh"
#include "scdm_rounds.cuh"

namespace lace {

namespace {

constexpr int QR_THREADS = 256;
constexpr int QR_MAXROWS = 1024;

struct Best {
    double v;
    int idx;
};

__device__ __forceinline__ bool better(double v, int i, double bv, int bi) { return v > bv || (v == bv && i < bi); }

// One column per thread: apply the previous reflection-free MGS step
// R[:,c] -= q (q . R[:,c]), then the exact squared norm of the column.
// Chosen columns report -1.  Per-block argmax (ties: lowest index).
template <typename T>
__global__ void __launch_bounds__(QR_THREADS) qr_update_kernel(int nrow, int ncol, T* __restrict__ R, size_t ld,
                                                               const T* __restrict__ q, int has_q,
                                                               const unsigned char* __restrict__ chosen,
                                                               Best* __restrict__ block_best) {
    __shared__ T qs[QR_MAXROWS];
    __shared__ double bv[QR_THREADS];
    __shared__ int bi[QR_THREADS];
    for (int r = threadIdx.x; r < nrow; r += blockDim.x) qs[r] = has_q ? q[r] : T(0);
    __syncthreads();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    double best = -2.0;
    int bidx = 0x7fffffff;
    if (c < ncol) {
        T* col = R + c;
        if (has_q) {
            T dot = T(0);
            for (int r = 0; r < nrow; ++r) dot += qs[r] * col[(size_t)r * ld];
            T nrm = T(0);
            for (int r = 0; r < nrow; ++r) {
                T v = col[(size_t)r * ld] - qs[r] * dot;
                col[(size_t)r * ld] = v;
                nrm += v * v;
            }
            best = chosen[c] ? -1.0 : (double)nrm;
        } else {
            T nrm = T(0);
            for (int r = 0; r < nrow; ++r) {
                T v = col[(size_t)r * ld];
                nrm += v * v;
            }
            best = chosen[c] ? -1.0 : (double)nrm;
        }
        bidx = c;
    }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = bidx;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            if (better(bv[threadIdx.x + o], bi[threadIdx.x + o], bv[threadIdx.x], bi[threadIdx.x])) {
                bv[threadIdx.x] = bv[threadIdx.x + o];
                bi[threadIdx.x] = bi[threadIdx.x + o];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) block_best[blockIdx.x] = Best{bv[0], bi[0]};
}

// Pick the pivot among the block winners, mark it, form q = R[:,p]/||R[:,p]||.
template <typename T>
__global__ void __launch_bounds__(QR_THREADS) qr_select_kernel(int nrow, int nblocks, const T* __restrict__ R,
                                                               size_t ld, const Best* __restrict__ block_best,
                                                               unsigned char* __restrict__ chosen, T* __restrict__ q,
                                                               int* __restrict__ piv, int step) {
    __shared__ double bv[QR_THREADS];
    __shared__ int bi[QR_THREADS];
    __shared__ double nrm_sh[QR_THREADS];
    double best = -3.0;
    int bidx = 0x7fffffff;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        const Best x = block_best[b];
        if (better(x.v, x.idx, best, bidx)) { best = x.v; bidx = x.idx; }
    }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = bidx;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o && better(bv[threadIdx.x + o], bi[threadIdx.x + o], bv[threadIdx.x], bi[threadIdx.x])) {
            bv[threadIdx.x] = bv[threadIdx.x + o];
            bi[threadIdx.x] = bi[threadIdx.x + o];
        }
        __syncthreads();
    }
    const int p = bi[0];
    double s = 0.0;
    for (int r = threadIdx.x; r < nrow; r += blockDim.x) {
        const double v = (double)R[(size_t)r * ld + p];
        s += v * v;
    }
    nrm_sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) nrm_sh[threadIdx.x] += nrm_sh[threadIdx.x + o];
        __syncthreads();
    }
    const double inv = nrm_sh[0] > 0.0 ? 1.0 / sqrt(nrm_sh[0]) : 0.0;
    for (int r = threadIdx.x; r < nrow; r += blockDim.x) q[r] = (T)((double)R[(size_t)r * ld + p] * inv);
    if (threadIdx.x == 0) {
        piv[step] = p;
        chosen[p] = 1;
    }
}

// Persistent pivoted QR in FP64: one cooperative launch runs every step, one CTA of
// 512 threads (16 warps) per SM.  A group of wpt warps owns 32-column tiles
// (lane = column); warp w of the group holds rows w*RPW .. w*RPW+RPW-1 of a
// tile.  The first nsm tiles of a group stay in shared memory across the steps,
// and only the rest is streamed from and back to global memory every step.  A
// step forms q.r (partial sums exchanged through shared memory behind the
// group's named barrier), updates the column, forms its exact new norm and the
// group's argmax; each CTA then publishes its best column's values, so one
// grid-wide barrier per step suffices: after it, every CTA picks the global
// winner and reads the winner's published column as the next q.  Block winners
// and published columns are double-buffered by step parity.
constexpr int QC_THREADS = 512, QC_WARPS = 16, RPW = 32, QC_MAXROWS = QC_WARPS * RPW;
static_assert(QC_MAXROWS <= QC_THREADS, "a published row a thread");

__device__ __forceinline__ void best_merge(double& v, int& i, double v2, int i2) {
    if (better(v2, i2, v, i)) { v = v2; i = i2; }
}

struct Vec4 {
    double a, b, c, d;
};
// four consecutive shared-memory values as 16-byte loads (16-byte aligned p)
__device__ __forceinline__ Vec4 load4(const double* p) {
    const double2 v0 = *reinterpret_cast<const double2*>(p), v1 = *reinterpret_cast<const double2*>(p + 2);
    return {v0.x, v0.y, v1.x, v1.y};
}

__device__ __forceinline__ void group_bar(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// q . v over this warp's RPW rows, four independent partial sums
__device__ __forceinline__ double dot_rows(const double* v, const double* qs, int rbase) {
    double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
#pragma unroll
    for (int j = 0; j < RPW; j += 4) {
        const Vec4 q4 = load4(qs + rbase + j);
        p0 += q4.a * v[j];
        p1 += q4.b * v[j + 1];
        p2 += q4.c * v[j + 2];
        p3 += q4.d * v[j + 3];
    }
    return (p0 + p1) + (p2 + p3);
}

// v -= q dot over the warp's rows, and the new squared norm of v
__device__ __forceinline__ double update_rows(double* v, const double* qs, int rbase, double dot) {
    double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;
#pragma unroll
    for (int j = 0; j < RPW; j += 4) {
        const Vec4 q4 = load4(qs + rbase + j);
        v[j] -= q4.a * dot;
        v[j + 1] -= q4.b * dot;
        v[j + 2] -= q4.c * dot;
        v[j + 3] -= q4.d * dot;
        n0 += v[j] * v[j];
        n1 += v[j + 1] * v[j + 1];
        n2 += v[j + 2] * v[j + 2];
        n3 += v[j + 3] * v[j + 3];
    }
    return (n0 + n1) + (n2 + n3);
}

__device__ __forceinline__ double norm_rows(const double* v) {
    double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;
#pragma unroll
    for (int j = 0; j < RPW; j += 4) {
        n0 += v[j] * v[j];
        n1 += v[j + 1] * v[j + 1];
        n2 += v[j + 2] * v[j + 2];
        n3 += v[j + 3] * v[j + 3];
    }
    return (n0 + n1) + (n2 + n3);
}

// Warp argmax of the 32 columns of a tile (lane = column), merged into (best, bidx).
__device__ __forceinline__ void tile_argmax(double cv, int ci, double& best, int& bidx) {
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, cv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, ci, o);
        best_merge(cv, ci, ov, oi);
    }
    best_merge(best, bidx, cv, ci);
}

__global__ void __launch_bounds__(QC_THREADS, 1)
    qr_persistent_kernel(int nrow, int ncol, double* __restrict__ R, int npiv, int wpt, int nsm,
                         Best* __restrict__ block_best, double* __restrict__ pub, unsigned char* __restrict__ chosen,
                         int* __restrict__ piv, unsigned* bar, unsigned long long limit_ns) {
    extern __shared__ __align__(16) unsigned char qr_smem_raw[];
    const int ngroups = QC_WARPS / wpt;
    double* stiles = reinterpret_cast<double*>(qr_smem_raw);  // [ngroups][nsm][wpt][RPW][32]
    double* pdot = stiles + (size_t)ngroups * nsm * wpt * RPW * 32;  // [nsm][QC_WARPS][32]
    double* pnrm = pdot + (size_t)nsm * QC_WARPS * 32;            // [nsm][QC_WARPS][32]
    __shared__ __align__(16) double qs[QC_MAXROWS + RPW];
    __shared__ double part[QC_WARPS * 32];
    __shared__ double gv[QC_WARPS];
    __shared__ int gi[QC_WARPS];
    __shared__ int wsel[QC_WARPS];
    __shared__ double red[QC_WARPS];
    __shared__ int pivot_sh, winner_sh, mybest_sh;
    __shared__ int abort_sh;
    unsigned gen = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = warp / wpt, wig = warp % wpt;
    const int ntiles = (ncol + 31) / 32;
    const int ggroup = blockIdx.x * ngroups + group, total_groups = gridDim.x * ngroups;
    const int ktot = ggroup < ntiles ? (ntiles - ggroup + total_groups - 1) / total_groups : 0;
    const int kres = min(ktot, nsm);  // this group's resident tiles
    const int rbase = wig * RPW;
    const int rows_pad = wpt * RPW;
    // chosen columns among this lane's resident tiles (bit k: resident tile k),
    // kept in a register so that a step reads no global flag for them
    unsigned cmask = 0u;
    for (int r = threadIdx.x; r < QC_MAXROWS + RPW; r += blockDim.x) qs[r] = 0.0;
    __syncthreads();
    for (int step = 0; step < npiv; ++step) {
        double best = -2.0;
        int bidx = 0x7fffffff;
        // resident tiles: all dot partials, one barrier, all updates and norm
        // partials, one barrier, then the argmax over the tiles
        if (step == 0) {
            for (int k = 0; k < kres; ++k) {
                const int c = (ggroup + k * total_groups) * 32 + lane;
                double* st = stiles + ((((size_t)group * nsm + k) * wpt + wig) * RPW) * 32 + lane;
                double v[RPW];
#pragma unroll
                for (int j = 0; j < RPW; ++j) {
                    v[j] = (c < ncol && rbase + j < nrow) ? R[(size_t)(rbase + j) * ncol + c] : 0.0;
                    st[j * 32] = v[j];
                }
                pnrm[(k * QC_WARPS + warp) * 32 + lane] = norm_rows(v);
            }
        } else {
            for (int k = 0; k < kres; ++k) {
                const double* st = stiles + ((((size_t)group * nsm + k) * wpt + wig) * RPW) * 32 + lane;
                double v[RPW];
#pragma unroll
                for (int j = 0; j < RPW; ++j) v[j] = st[j * 32];
                pdot[(k * QC_WARPS + warp) * 32 + lane] = dot_rows(v, qs, rbase);
            }
            if (kres > 0) group_bar(1 + group, wpt * 32);
            for (int k = 0; k < kres; ++k) {
                double* st = stiles + ((((size_t)group * nsm + k) * wpt + wig) * RPW) * 32 + lane;
                double dot = 0.0;
                for (int w = 0; w < wpt; ++w) dot += pdot[(k * QC_WARPS + group * wpt + w) * 32 + lane];
                double v[RPW];
#pragma unroll
                for (int j = 0; j < RPW; ++j) v[j] = st[j * 32];
                pnrm[(k * QC_WARPS + warp) * 32 + lane] = update_rows(v, qs, rbase, dot);
#pragma unroll
                for (int j = 0; j < RPW; ++j) st[j * 32] = v[j];
            }
        }
        if (kres > 0) group_bar(1 + group, wpt * 32);
        if (wig == 0) {
            for (int k = 0; k < kres; ++k) {
                double tot = 0.0;
                for (int w = 0; w < wpt; ++w) tot += pnrm[(k * QC_WARPS + group * wpt + w) * 32 + lane];
                const int c = (ggroup + k * total_groups) * 32 + lane;
                const bool live = c < ncol && !((cmask >> k) & 1u);
                tile_argmax(live ? (double)tot : (c < ncol ? -1.0 : -2.0), c < ncol ? c : 0x7fffffff, best, bidx);
            }
        }
        // the rest: streamed from and back to global memory, one tile at a time
        for (int tile = ggroup + nsm * total_groups; tile < ntiles; tile += total_groups) {
            const int c = tile * 32 + lane;
            const bool live = c < ncol && !chosen[c];
            double v[RPW];
            const bool full = rbase + RPW <= nrow;
            if (full) {
#pragma unroll
                for (int j = 0; j < RPW; ++j) v[j] = live ? R[(size_t)(rbase + j) * ncol + c] : 0.0;
            } else {
#pragma unroll
                for (int j = 0; j < RPW; ++j)
                    v[j] = (live && rbase + j < nrow) ? R[(size_t)(rbase + j) * ncol + c] : 0.0;
            }
            if (step > 0) {
                part[warp * 32 + lane] = dot_rows(v, qs, rbase);
                group_bar(1 + group, wpt * 32);
                double dot = 0.0;
                for (int w = 0; w < wpt; ++w) dot += part[(group * wpt + w) * 32 + lane];
                group_bar(1 + group, wpt * 32);
                part[warp * 32 + lane] = update_rows(v, qs, rbase, dot);
                if (live) {
                    if (full) {
#pragma unroll
                        for (int j = 0; j < RPW; ++j) R[(size_t)(rbase + j) * ncol + c] = v[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < RPW; ++j)
                            if (rbase + j < nrow) R[(size_t)(rbase + j) * ncol + c] = v[j];
                    }
                }
            } else {
                part[warp * 32 + lane] = norm_rows(v);
            }
            group_bar(1 + group, wpt * 32);
            if (wig == 0) {
                double tot = 0.0;
                for (int w = 0; w < wpt; ++w) tot += part[(group * wpt + w) * 32 + lane];
                tile_argmax(live ? (double)tot : (c < ncol ? -1.0 : -2.0), c < ncol ? c : 0x7fffffff, best, bidx);
            }
            group_bar(1 + group, wpt * 32);
        }
        if (lane == 0 && wig == 0) { gv[group] = best; gi[group] = bidx; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double b = gv[0];
            int bi_ = gi[0];
            for (int w = 1; w < ngroups; ++w) best_merge(b, bi_, gv[w], gi[w]);
            block_best[(step & 1) * gridDim.x + blockIdx.x] = Best{b, bi_};
            mybest_sh = (b >= 0.0 && bi_ < ncol) ? bi_ : -1;
        }
        __syncthreads();
        // publish this CTA's candidate column (its current residual values) and,
        // in slot rows_pad, the inverse of its FP64 norm
        {
            double* out = pub + ((size_t)(step & 1) * gridDim.x + blockIdx.x) * (rows_pad + 4);
            const int cb = mybest_sh;
            if (cb >= 0) {
                const int tile = cb / 32, cl = cb % 32;
                const int kk = tile / total_groups, gg = tile % total_groups - blockIdx.x * ngroups;
                double x = 0.0;
                if (kk < nsm) {
                    const double* st = stiles + (((size_t)gg * nsm + kk) * wpt) * RPW * 32 + cl;
                    if (threadIdx.x < rows_pad) {
                        x = st[(size_t)threadIdx.x * 32];
                        out[threadIdx.x] = x;
                    }
                } else {
                    if (threadIdx.x < rows_pad) {
                        x = threadIdx.x < nrow ? R[(size_t)threadIdx.x * ncol + cb] : 0.0;
                        out[threadIdx.x] = x;
                    }
                }
                double s2 = x * x;
                for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
                if (lane == 0) red[warp] = s2;
                __syncthreads();
                if (threadIdx.x == 0) {
                    double t = 0.0;
                    for (int w = 0; w < QC_WARPS; ++w) t += red[w];
                    out[rows_pad] = t > 0.0 ? 1.0 / sqrt(t) : 0.0;
                }
            }
        }
        if (!grid_barrier(bar, gen, &abort_sh, limit_ns)) return;
        // every CTA: global argmax (one block winner per thread: a single round
        // of loads), then q = (winner's column) x (its inverse norm)
        {
            double gb = -3.0;
            int gbi = 0x7fffffff, gw = 0;
            if (threadIdx.x < gridDim.x) {
                const Best x = block_best[(step & 1) * gridDim.x + threadIdx.x];
                gb = x.v;
                gbi = x.idx;
                gw = threadIdx.x;
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, gb, o);
                const int oi = __shfl_xor_sync(0xffffffffu, gbi, o);
                const int ow = __shfl_xor_sync(0xffffffffu, gw, o);
                if (better(ov, oi, gb, gbi)) { gb = ov; gbi = oi; gw = ow; }
            }
            if (lane == 0) { gv[warp] = gb; gi[warp] = gbi; wsel[warp] = gw; }
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < QC_WARPS; ++w)
                    if (better(gv[w], gi[w], gb, gbi)) { gb = gv[w]; gbi = gi[w]; gw = wsel[w]; }
                pivot_sh = gbi;
                winner_sh = gw;
            }
        }
        __syncthreads();
        const int p = pivot_sh;
        {
            const double* col = pub + ((size_t)(step & 1) * gridDim.x + winner_sh) * (rows_pad + 4);
            const double inv = (double)col[rows_pad];
            for (int r = threadIdx.x; r < nrow; r += blockDim.x) qs[r] = col[r] * inv;
        }
        if (threadIdx.x == 0) {
            chosen[p] = 1;
            if (blockIdx.x == 0) piv[step] = p;
        }
        {
            const int tile = p / 32, gg = tile % total_groups, kk = tile / total_groups;
            if (gg / ngroups == (int)blockIdx.x && group == gg % ngroups && lane == p % 32 && kk < nsm)
                cmask |= 1u << kk;
        }
        __syncthreads();
    }
}

template <typename T>
__global__ void gather_subsample_kernel(int n1, int n2, int n3, int stride, int m1, int m2, int m3,
                                        const T* __restrict__ psi, size_t ng, T* __restrict__ out, size_t ncol) {
    const int o = blockIdx.y;
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncol; c += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(c % m3);
        const int j = (int)((c / m3) % m2);
        const int i = (int)(c / ((size_t)m3 * m2));
        const size_t full = ((size_t)(i * stride) * n2 + (size_t)(j * stride)) * n3 + (size_t)(k * stride);
        out[(size_t)o * ncol + c] = psi[(size_t)o * ng + full];
    }
    (void)n1;
    (void)m1;
}

template <typename T>
__global__ void gather_columns_kernel(const T* __restrict__ psi, size_t ldpsi, int norb,
                                      const long long* __restrict__ idx, int npts, double* __restrict__ out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= npts * norb) return;
    const int p = e / norb, o = e % norb;
    out[e] = (double)psi[(size_t)o * ldpsi + (size_t)idx[p]];
}

// Thread i: grid point of pivot i and its rank among all by the Z-order code
// (coordinate bits interleaved), codes recomputed 256 at a time in shared
// memory.
__global__ void __launch_bounds__(256) pivot_points_kernel(int n1, int n2, int m1, int m2, int m3, int stride, int n,
                                                           const int* __restrict__ piv, long long* __restrict__ full,
                                                           int* __restrict__ order) {
    __shared__ unsigned long long code[256];
    auto spread = [](unsigned long long v) {  // two zero bits between 21 bits
        v &= 0x1fffff;
        v = (v | v << 32) & 0x1f00000000ffffULL;
        v = (v | v << 16) & 0x1f0000ff0000ffULL;
        v = (v | v << 8) & 0x100f00f00f00f00fULL;
        v = (v | v << 4) & 0x10c30c30c30c30c3ULL;
        return (v | v << 2) & 0x1249249249249249ULL;
    };
    auto point = [&](int k) -> long long {
        if (!piv) return full[k];
        const int c = min(max(piv[k], 0), m1 * m2 * m3 - 1);  // (invalid after a timeout)
        return ((long long)(c / (m3 * m2) * stride) * n1 + (long long)(c / m3 % m2) * stride) * n2 + (long long)(c % m3) * stride;
    };
    auto code_of = [&](long long p) {
        return spread((unsigned long long)(p / ((long long)n2 * n1))) << 2 | spread((unsigned long long)(p / n2 % n1)) << 1 |
               spread((unsigned long long)(p % n2));
    };
    const int i = blockIdx.x * 256 + threadIdx.x;
    const long long mine = i < n ? point(i) : 0;
    const unsigned long long c = code_of(mine);
    int rank = 0;
    for (int j0 = 0; j0 < n; j0 += 256) {
        __syncthreads();
        if (j0 + (int)threadIdx.x < n) code[threadIdx.x] = code_of(point(j0 + threadIdx.x));
        __syncthreads();
        const int m = min(256, n - j0);
        for (int j = 0; j < m; ++j) rank += code[j] < c || (code[j] == c && j0 + j < i);
    }
    if (i < n) {
        if (piv) full[i] = mine;
        order[rank] = i;
    }
}

}  // namespace

static size_t align256(size_t b) { return (b + 255) / 256 * 256; }

// Capacity (in Best entries) of the block-winner buffer of qrcp_aux_bytes.
static int nblocks_cap(int ncol) { return std::max((ncol + QR_THREADS - 1) / QR_THREADS, 2 * 152 * 8); }

// Published candidate columns of the persistent FP64 kernel: 2 (step parity) x
// CTAs (up to 304) x padded rows (< 2 nrow + 64).
static size_t pub_bytes(int nrow) { return align256((size_t)2 * 304 * (2 * (size_t)nrow + 64) * sizeof(double)); }

size_t qrcp_aux_bytes(int nrow, int ncol) {
    const int nblocks = nblocks_cap(ncol);
    return align256(sizeof(Best) * nblocks) + align256((size_t)ncol) + align256(sizeof(double) * nrow) + 256 +
           std::max(pub_bytes(nrow), qrr::buf_bytes(nrow, ncol));
}

// The persistent FP64 kernel; *ran = false when the rows do not fit its warp layout
// or the device cannot co-schedule it.
static cudaError_t qr_persistent_launch(int nrow, int ncol, double* R, int npiv, Best* best, double* pub,
                                        unsigned char* chosen, int* d_piv, unsigned* bar,
                                        unsigned long long limit_ns, cudaStream_t s, int* launches, bool* ran) {
    *ran = false;
    int dev = 0, sms = 0, coop = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int wpt = 2;  // >= 2 keeps the named-barrier ids (1 + group) within 1..8
    while (wpt * RPW < nrow) wpt *= 2;
    if (!coop || wpt > QC_WARPS || nrow > QC_MAXROWS || sms > 304 || 2 * sms > nblocks_cap(ncol) ||
        (size_t)2 * sms * (wpt * RPW + 4) * sizeof(double) > pub_bytes(nrow))
        return cudaSuccess;
    const void* fn = (const void*)qr_persistent_kernel;
    cudaFuncAttributes fa{};
    cudaError_t e;
    if ((e = cudaFuncGetAttributes(&fa, fn))) return e;
    // one limit for every caller of this kernel: the opt-in maximum
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes)))
        return e;
    const int ngroups = QC_WARPS / wpt;
    const int ntiles = (ncol + 31) / 32;
    // no more CTAs than tiles: a small matrix then syncs fewer CTAs per step and
    // leaves SMs to other work
    const int ctas = std::min(sms, std::max(1, (ntiles + ngroups - 1) / ngroups));
    const int total_groups = ctas * ngroups;
    const int max_k = (ntiles + total_groups - 1) / total_groups;
    const size_t tile_bytes = (size_t)wpt * RPW * 32 * sizeof(double);  // one tile slot of one group
    const size_t red_bytes = (size_t)2 * QC_WARPS * 32 * sizeof(double);  // dot and norm partials of one tile slot
    const size_t budget = (size_t)std::max(0, optin - (int)fa.sharedSizeBytes - 1024);
    int nsm = (int)std::min<size_t>((size_t)max_k, budget / (ngroups * tile_bytes + red_bytes));
    nsm = std::min(nsm, 30);  // the per-lane chosen mask has 32 bits
    const size_t dyn = (size_t)ngroups * nsm * tile_bytes + (size_t)nsm * red_bytes;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, QC_THREADS, dyn))) return e;
    if (per_sm < 1) return cudaSuccess;
    if ((e = cudaMemsetAsync(bar, 0, 4 * sizeof(unsigned), s))) return e;
    void* args[] = {(void*)&nrow, (void*)&ncol, (void*)&R,   (void*)&npiv,   (void*)&wpt,  (void*)&nsm,
                    (void*)&best, (void*)&pub,  (void*)&chosen, (void*)&d_piv, (void*)&bar, (void*)&limit_ns};
    if ((e = cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(QC_THREADS), args, dyn, s))) return e;
    *launches += 1;
    *ran = true;
    return cudaSuccess;
}

// The pivoted QR in rounds (scdm_rounds.cuh); *ran = false when the device
// cannot co-schedule its CTAs.
template <int NRL>
static cudaError_t qr_rounds_launch(int nrow, int ncol, const float* R, int npiv, void* aux, int* d_piv, unsigned* bar,
                                    unsigned long long limit_ns, cudaStream_t s, int* launches, bool* ran) {
    *ran = false;
    int dev = 0, sms = 0, coop = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const void* fn = (const void*)qrr::rounds_kernel<NRL>;
    cudaFuncAttributes fa{};
    cudaError_t e;
    if ((e = cudaFuncGetAttributes(&fa, fn))) return e;
    const size_t dyn = qrr::smem_bytes();
    if (!coop || nrow > 32 * NRL || npiv > nrow || dyn + fa.sharedSizeBytes + 1024 > (size_t)optin) return cudaSuccess;
    // one limit for every caller of this kernel: the opt-in maximum
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes)))
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, qrr::kThreads, dyn))) return e;
    if (per_sm < 1) return cudaSuccess;
    const int ctas = std::min(sms, (ncol + qrr::kTile - 1) / qrr::kTile);
    qrr::Buf B = qrr::buf_at(aux, nrow, ncol);
    if ((e = cudaMemsetAsync(bar, 0, 4 * sizeof(unsigned), s))) return e;
    if ((e = cudaMemsetAsync(B.hist, 0, sizeof(unsigned) * qrr::kBins, s))) return e;
    if ((e = cudaMemsetAsync(B.ctl, 0, 16 * sizeof(unsigned), s))) return e;
    if ((e = cudaMemsetAsync(B.ctl + 4, 0xff, 2 * sizeof(unsigned), s))) return e;
    void* args[] = {(void*)&nrow, (void*)&ncol, (void*)&R, (void*)&npiv, (void*)&B, (void*)&d_piv, (void*)&bar, (void*)&limit_ns};
    if ((e = cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(qrr::kThreads), args, dyn, s))) return e;
    *launches += 1;
    *ran = true;
    return cudaSuccess;
}

// R (nrow x ncol, row-major, leading dimension ncol) may be overwritten.  aux is
// caller-provided scratch of qrcp_aux_bytes(nrow, ncol) bytes.
template <typename T>
cudaError_t qrcp_pivots(int nrow, int ncol, T* R, int npiv, int* d_piv, void* aux, int* h_timeout,
                        unsigned long long wait_limit_ns, cudaStream_t s, int* launches) {
    *h_timeout = 0;
    if (nrow > QR_MAXROWS || npiv > ncol) return cudaErrorInvalidValue;
    const int nblocks = (ncol + QR_THREADS - 1) / QR_THREADS;
    unsigned char* base = static_cast<unsigned char*>(aux);
    Best* best = reinterpret_cast<Best*>(base);
    unsigned char* chosen = base + align256(sizeof(Best) * nblocks_cap(ncol));
    T* q = reinterpret_cast<T*>(chosen + align256((size_t)ncol));
    unsigned* bar = reinterpret_cast<unsigned*>(reinterpret_cast<unsigned char*>(q) + align256(sizeof(double) * nrow));
    T* pub = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(bar) + 256);
    cudaMemsetAsync(chosen, 0, ncol, s);
    // cooperative versions: in rounds (FP32), a barrier a pivot (FP64)
    bool ran = false;
    cudaError_t e;
    if constexpr (sizeof(T) == 4) {
        // At 72^3 with 256 orbitals 0.67 ms (one barrier a pivot with the matrix
        // in registers and shared memory: 2.37 ms), at 120^3 with 320, off chip,
        // 1.7 ms (73.4 ms); 16 orbitals on 32^3 take the same time either way.
        auto go = [&](auto launch) {
            return launch(nrow, ncol, R, npiv, reinterpret_cast<unsigned char*>(bar) + 256, d_piv, bar, wait_limit_ns, s,
                          launches, &ran);
        };
        e = nrow <= 256 ? go(qr_rounds_launch<8>) : nrow <= 512 ? go(qr_rounds_launch<16>) : go(qr_rounds_launch<32>);
    } else {
        e = qr_persistent_launch(nrow, ncol, R, npiv, best, pub, chosen, d_piv, bar, wait_limit_ns, s, launches, &ran);
    }
    if (e) return e;
    if (ran) {
        return cudaMemcpyAsync(h_timeout, bar + 2, sizeof(int), cudaMemcpyDeviceToHost, s);
    }
    for (int step = 0; step < npiv; ++step) {
        qr_update_kernel<T><<<nblocks, QR_THREADS, 0, s>>>(nrow, ncol, R, (size_t)ncol, q, step > 0, chosen, best);
        qr_select_kernel<T><<<1, QR_THREADS, 0, s>>>(nrow, nblocks, R, (size_t)ncol, best, chosen, q, d_piv, step);
        *launches += 2;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t gather_subsample(const GridGeom& g, int stride, const T* psi, int norb, T* out, int* ncol_out,
                             cudaStream_t s, int* launches) {
    const int m1 = (g.n[0] + stride - 1) / stride, m2 = (g.n[1] + stride - 1) / stride,
              m3 = (g.n[2] + stride - 1) / stride;
    const size_t ncol = (size_t)m1 * m2 * m3;
    *ncol_out = (int)ncol;
    dim3 grid((unsigned)std::min<size_t>((ncol + 255) / 256, 1024), norb);
    gather_subsample_kernel<T><<<grid, 256, 0, s>>>(g.n[0], g.n[1], g.n[2], stride, m1, m2, m3, psi, g.ng, out, ncol);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t pivot_points(const GridGeom& g, int stride, int n, const int* piv, long long* full, int* order, cudaStream_t s,
                         int* launches) {
    const int m1 = (g.n[0] + stride - 1) / stride, m2 = (g.n[1] + stride - 1) / stride,
              m3 = (g.n[2] + stride - 1) / stride;
    pivot_points_kernel<<<(n + 255) / 256, 256, 0, s>>>(g.n[1], g.n[2], m1, m2, m3, stride, n, piv, full, order);
    *launches += 1;
    return cudaGetLastError();
}

template <typename T>
cudaError_t gather_columns(const T* psi, size_t ldpsi, int norb, const long long* d_full_idx, int npts, double* out,
                           cudaStream_t s, int* launches) {
    const int tot = npts * norb;
    gather_columns_kernel<T><<<(tot + 255) / 256, 256, 0, s>>>(psi, ldpsi, norb, d_full_idx, npts, out);
    *launches += 1;
    return cudaGetLastError();
}

template cudaError_t qrcp_pivots<float>(int, int, float*, int, int*, void*, int*, unsigned long long, cudaStream_t,
                                         int*);
template cudaError_t qrcp_pivots<double>(int, int, double*, int, int*, void*, int*, unsigned long long, cudaStream_t,
                                          int*);
template cudaError_t gather_subsample<float>(const GridGeom&, int, const float*, int, float*, int*, cudaStream_t, int*);
template cudaError_t gather_subsample<double>(const GridGeom&, int, const double*, int, double*, int*, cudaStream_t,
                                              int*);
template cudaError_t gather_columns<float>(const float*, size_t, int, const long long*, int, double*, cudaStream_t,
                                           int*);
template cudaError_t gather_columns<double>(const double*, size_t, int, const long long*, int, double*, cudaStream_t,
                                            int*);

}  // namespace lace
