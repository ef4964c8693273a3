// p2g_chunks_16.cu -- the P2G chunk kernels for 16-bit coefficient codes, 27 modes.
#include "p2g_chunks.cuh"

namespace polypic {

cudaError_t launch_chunks_16(const P2GArgs &P, int fmt, int grid, cudaStream_t s) {
    if (fmt == POLYPIC_COEFF_BF16) return launch_chunks<27, POLYPIC_COEFF_BF16, false>(P, grid, s);
    if (fmt == POLYPIC_COEFF_F16) return launch_chunks<27, POLYPIC_COEFF_F16, false>(P, grid, s);
    return cudaErrorInvalidValue;
}

}  // namespace polypic
