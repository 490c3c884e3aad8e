// Lane passes of the pair convolutions (pairconv_lanes.cuh): passes A and C of the cubes 48^3, 50^3, 54^3, 60^3.
#include "pairconv_lanes.cuh"

namespace lace {
namespace ln {

bool cube_2(int n, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    switch (n) {
        case 48: return launch_cube<48>(pass, nb, P, g0, s);
        case 50: return launch_cube<50>(pass, nb, P, g0, s);
        case 54: return launch_cube<54>(pass, nb, P, g0, s);
        case 60: return launch_cube<60>(pass, nb, P, g0, s);
        default: return false;
    }
}

}  // namespace ln
}  // namespace lace
