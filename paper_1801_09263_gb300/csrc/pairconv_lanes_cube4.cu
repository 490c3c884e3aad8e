// Lane passes of the pair convolutions (pairconv_lanes.cuh): passes A and C of the cubes 96^3, 100^3, 108^3, 120^3, 128^3.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool cube_4(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 96: return launch_cube<96>(pass, nb, P, g0, s);
        case 100: return launch_cube<100>(pass, nb, P, g0, s);
        case 108: return launch_cube<108>(pass, nb, P, g0, s);
        case 120: return launch_cube<120>(pass, nb, P, g0, s);
        case 128: return launch_cube<128>(pass, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
