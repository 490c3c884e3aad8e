// Lane passes of the pair convolutions (pairconv_lanes.cuh): pass B along x axes of 80, 81, 90, 96, 100, 108, 120, 128 points.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool slab_3(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 80: return launch_slab<80>(M, nb, P, g0, s);
        case 81: return launch_slab<81>(M, nb, P, g0, s);
        case 90: return launch_slab<90>(M, nb, P, g0, s);
        case 96: return launch_slab<96>(M, nb, P, g0, s);
        case 100: return launch_slab<100>(M, nb, P, g0, s);
        case 108: return launch_slab<108>(M, nb, P, g0, s);
        case 120: return launch_slab<120>(M, nb, P, g0, s);
        case 128: return launch_slab<128>(M, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
