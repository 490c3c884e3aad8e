// Sum over the K chunks of a Gram, FP64 in a fixed order.
#pragma once

#include <cuda_runtime.h>

namespace lace {
namespace {

constexpr int kSumWarps = 8;

// 32 consecutive outputs a block, its warps each an eighth of the chunks: reads
// stay coalesced and an output's chunks are in flight together.  256 x 64 outputs
// of 76 chunks took 14 us with a warp an output (a sector for every value) and
// longer with a thread an output (one chunk after the other).  tile: rows of the
// tiles of a symmetric product, of which only those on and above the diagonal hold
// values; the rest is read mirrored.
__global__ void __launch_bounds__(32 * kSumWarps) chunk_sum_kernel(int M, int N, int nchunk, const double* __restrict__ work,
                                                                   double alpha, bool sym, int tile, double* __restrict__ C,
                                                                   int ldc) {
    __shared__ double part[kSumWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t tot = (size_t)M * N, idx = (size_t)blockIdx.x * 32 + lane;
    const int m = (int)(idx / N), n = (int)(idx % N);
    double s = 0.0;
    if (idx < tot) {
        const double* src = work + ((sym && n / tile < m / tile) ? (size_t)n * N + m : idx);
#pragma unroll 4
        for (int c = warp; c < nchunk; c += kSumWarps) s += src[(size_t)c * tot];
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp > 0 || idx >= tot) return;
#pragma unroll
    for (int w = 1; w < kSumWarps; ++w) s += part[w][lane];
    C[(size_t)m * ldc + n] = alpha * s;
}

// Returns the error of its own launch or of one before it (reading clears it, so the
// caller has to pass it on).
[[nodiscard]] cudaError_t chunk_sum(int M, int N, size_t nchunk, const double* work, double alpha, bool sym, int tile, double* C,
                                    int ldc, cudaStream_t s) {
    chunk_sum_kernel<<<(unsigned)(((size_t)M * N + 31) / 32), 32 * kSumWarps, 0, s>>>(M, N, (int)nchunk, work, alpha, sym, tile,
                                                                                      C, ldc);
    return cudaGetLastError();
}

}  // namespace
}  // namespace lace
