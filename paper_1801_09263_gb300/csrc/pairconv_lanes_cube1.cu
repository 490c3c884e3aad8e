// Lane passes of the pair convolutions (pairconv_lanes.cuh): passes A and C of the cubes 24^3, 30^3, 32^3, 36^3, 40^3.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool cube_1(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 24: return launch_cube<24>(pass, nb, P, g0, s);
        case 30: return launch_cube<30>(pass, nb, P, g0, s);
        case 32: return launch_cube<32>(pass, nb, P, g0, s);
        case 36: return launch_cube<36>(pass, nb, P, g0, s);
        case 40: return launch_cube<40>(pass, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
