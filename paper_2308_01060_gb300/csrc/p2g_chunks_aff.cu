// p2g_chunks_aff.cu -- the P2G chunk kernels of Eq 12's affine map with 8 and 27
// modes, evaluated per stencil node.
#include "p2g_chunks.cuh"

namespace polypic {

cudaError_t launch_chunks_aff(const P2GArgs &P, int R, int grid, cudaStream_t s) {
    if (R == 8) return launch_chunks<8, POLYPIC_COEFF_F32, false, true>(P, grid, s);
    if (R == 27) return launch_chunks<27, POLYPIC_COEFF_F32, false, true>(P, grid, s);
    return cudaErrorInvalidValue;
}

}  // namespace polypic
