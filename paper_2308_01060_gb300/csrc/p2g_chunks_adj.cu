// p2g_chunks_adj.cu -- the P2G chunk kernel of the G2P adjoint's scatter, 27 modes.
#include "p2g_chunks.cuh"

namespace polypic {

cudaError_t launch_chunks_adj(const P2GArgs &P, int grid, cudaStream_t s) {
    return launch_chunks<27, POLYPIC_COEFF_F32, true>(P, grid, s);
}

}  // namespace polypic
