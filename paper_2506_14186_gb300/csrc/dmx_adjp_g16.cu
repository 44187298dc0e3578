// Reverse-mode adjoint kernel with model-parameter gradients, 16 lanes per
// environment (one translation unit per lane count, as dmx_adj_g16.cu).
#include "dmx_adjoint_rev.cuh"

namespace dmx {
template cudaError_t launch_adjoint_rev_g<16, true, DevModel>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<16, true, DevModel>(int, size_t);
}  // namespace dmx
