// p2g_tiles_aff.cu -- the P2G tile kernel with Eq 12's affine map of 4 modes
// (FP32 coefficients).
#include "p2g_tiles.cuh"

namespace polypic {

cudaError_t launch_tiles_aff4(const P2GArgs &P, int grid, cudaStream_t s) {
    return launch_tiles<4, POLYPIC_COEFF_F32, false, true>(P, grid, s);
}

}  // namespace polypic
