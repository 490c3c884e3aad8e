// Lane passes of the pair convolutions (pairconv_lanes.cuh): pass B along x axes of 24, 25, 27, 30, 32, 36, 40, 45 points.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool slab_1(int n, int M, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 24: return launch_slab<24>(M, nb, P, g0, s);
        case 25: return launch_slab<25>(M, nb, P, g0, s);
        case 27: return launch_slab<27>(M, nb, P, g0, s);
        case 30: return launch_slab<30>(M, nb, P, g0, s);
        case 32: return launch_slab<32>(M, nb, P, g0, s);
        case 36: return launch_slab<36>(M, nb, P, g0, s);
        case 40: return launch_slab<40>(M, nb, P, g0, s);
        case 45: return launch_slab<45>(M, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
