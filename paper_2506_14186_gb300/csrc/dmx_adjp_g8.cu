// Reverse-mode adjoint kernel with model-parameter gradients, 8 lanes per
// environment (one translation unit per lane count, as dmx_adj_g8.cu).
#include "dmx_adjoint_rev.cuh"

namespace dmx {
template cudaError_t launch_adjoint_rev_g<8, true, DevModel>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<8, true, DevModel>(int, size_t);
}  // namespace dmx
