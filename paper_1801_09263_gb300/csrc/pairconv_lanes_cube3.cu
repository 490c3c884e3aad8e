// Lane passes of the pair convolutions (pairconv_lanes.cuh): passes A and C of the cubes 64^3, 72^3, 80^3, 90^3.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool cube_3(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 64: return launch_cube<64>(pass, nb, P, g0, s);
        case 72: return launch_cube<72>(pass, nb, P, g0, s);
        case 80: return launch_cube<80>(pass, nb, P, g0, s);
        case 90: return launch_cube<90>(pass, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
