// Lane passes of the pair convolutions (pairconv_lanes.cuh): pass B along x axes of 48, 50, 54, 60, 64, 72, 75 points.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool slab_2(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 48: return launch_slab<48>(M, nb, P, g0, s);
        case 50: return launch_slab<50>(M, nb, P, g0, s);
        case 54: return launch_slab<54>(M, nb, P, g0, s);
        case 60: return launch_slab<60>(M, nb, P, g0, s);
        case 64: return launch_slab<64>(M, nb, P, g0, s);
        case 72: return launch_slab<72>(M, nb, P, g0, s);
        case 75: return launch_slab<75>(M, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
