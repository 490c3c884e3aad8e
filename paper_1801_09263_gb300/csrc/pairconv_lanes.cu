// Lane passes of the pair convolutions (pairconv_lanes.cuh): the boxes, the
// table of K in the order of the passes, and the choice of the kernels.
#include "pairconv_box.cuh"

namespace lace {
namespace ln {

void box_pass(int n1, int n2, int n3, int pass, int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    static OncePerDevice once;
    once.run([&] {
        smem_opt_in(box_a<kBoxRegs>, plane_smem(kMaxN, kMaxN));
        smem_opt_in(box_c<kBoxRegs>, plane_smem(kMaxN, kMaxN));
    });
    const Box b = make_box(n2, n3);
    const size_t sm = plane_smem(n2, n3);
    const int nt = plane_threads(n2, n3);
    if (pass == 0) box_a<kBoxRegs><<<dim3(nb, n1), nt, sm, s>>>(P, g0, b);
    else box_c<kBoxRegs><<<dim3(nb, n1), nt, sm, s>>>(P, g0, b);
}

// out[sx][sy][c][lane] = -k[x][y][z] at the frequencies of the slots.
__global__ void klanes_kernel(const float* __restrict__ k, float* __restrict__ out, int n1, int n2, int n3, Radices rx,
                              Radices ry, Radices rz) {
    const int h = n3 / 2, c = blockIdx.x * blockDim.x + threadIdx.x, sy = blockIdx.y, sx = blockIdx.z;
    if (c >= h) return;
    const int x = slot_k(sx, rx.big, rx.small), y = slot_k(sy, ry.small, ry.big), z = slot_k(c, rz.big, rz.small);
    const float* row = k + ((size_t)x * n2 + y) * n3;
    reinterpret_cast<float2*>(out)[((size_t)sx * n2 + sy) * h + c] = make_float2(-row[z], -row[z + h]);
}

}  // namespace ln

// The lane passes take grids with an even z size whose axes (z: half of it)
// have two radices; 24 points an axis at least (smaller grids leave the
// choice without effect, and keep the generic passes).
bool lanes_ok(const int n[3]) {
    if (n[2] % 2) return false;
    for (int a = 0; a < 3; ++a)
        if (n[a] < 24 || n[a] > kMaxN) return false;
    return ln::radices(n[0]).big && ln::radices(n[1]).big && ln::radices(n[2] / 2).big;
}

cudaError_t lanes_ktab(const int n[3], const float* d_ktab, float* d_out, cudaStream_t s) {
    ln::klanes_kernel<<<dim3((n[2] / 2 + 31) / 32, n[1], n[0]), 32, 0, s>>>(d_ktab, d_out, n[0], n[1], n[2],
                                                                        ln::radices(n[0]), ln::radices(n[1]),
                                                                        ln::radices(n[2] / 2));
    return cudaGetLastError();
}

bool lanes_launch(const int n[3], int nb, const ConvArgs<float>& P, int g0, cudaStream_t s) {
    if (!lanes_ok(n)) return false;
    const bool cube = n[0] == n[1] && n[1] == n[2];
    auto plane = [&](int pass) {
        if (cube && (ln::cube_1(n[0], pass, nb, P, g0, s) || ln::cube_2(n[0], pass, nb, P, g0, s) ||
                     ln::cube_3(n[0], pass, nb, P, g0, s) || ln::cube_4(n[0], pass, nb, P, g0, s)))
            return;
        ln::box_pass(n[0], n[1], n[2], pass, nb, P, g0, s);
    };
    const int M = n[1] * (n[2] / 2);
    plane(0);
    if (!ln::slab_1(n[0], M, nb, P, g0, s) && !ln::slab_2(n[0], M, nb, P, g0, s) &&
        !ln::slab_3(n[0], M, nb, P, g0, s))
        return false;
    plane(2);
    return true;
}

}  // namespace lace
