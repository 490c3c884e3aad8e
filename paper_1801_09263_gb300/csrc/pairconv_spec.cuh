// Radix plans of the size-specialised FP32 pass bodies (pairconv_spec2.cuh):
// two register radices per axis, compile-time.
#pragma once

#include "lace_internal.cuh"

namespace lace {
namespace spec {

using C = float2;

struct Plan2 {
    int r1, r2;
};

__host__ __device__ constexpr bool radix_ok(int r) {
    return r == 2 || r == 3 || r == 4 || r == 5 || r == 6 || r == 8 || r == 9 || r == 10 || r == 12 || r == 16;
}

// Two register radices r1 * r2 = n with the largest smaller factor.
__host__ __device__ constexpr Plan2 plan2(int n) {
    Plan2 best{0, 0};
    int best_min = 0;
    for (int r1 = 16; r1 >= 2; --r1) {
        if (!radix_ok(r1) || n % r1) continue;
        const int r2 = n / r1;
        if (!radix_ok(r2)) continue;
        const int mn = r1 < r2 ? r1 : r2;
        if (mn > best_min) {
            best_min = mn;
            best = Plan2{r1, r2};
        }
    }
    return best;
}

__device__ __forceinline__ void kahan(float& s, float& c, float v) {
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

}  // namespace spec
}  // namespace lace
