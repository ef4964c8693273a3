// p2g_chunks_f32.cu -- the P2G chunk kernels for FP32 coefficients and the
// constant map: 27 modes, and solid phases of 4 and 8.
#include "p2g_chunks.cuh"

namespace polypic {

cudaError_t launch_chunks_f32(const P2GArgs &P, int R, int grid, cudaStream_t s) {
    if (R == 4) return launch_chunks<4, POLYPIC_COEFF_F32, false>(P, grid, s);
    if (R == 8) return launch_chunks<8, POLYPIC_COEFF_F32, false>(P, grid, s);
    if (R == 27) return launch_chunks<27, POLYPIC_COEFF_F32, false>(P, grid, s);
    return cudaErrorInvalidValue;
}

}  // namespace polypic
