// Reverse-mode adjoint kernel with model-parameter gradients, 32 lanes per
// environment (one translation unit per lane count, as dmx_adj_g32.cu).
#include "dmx_adjoint_rev.cuh"

namespace dmx {
template cudaError_t launch_adjoint_rev_g<32, true, DevModel>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<32, true, DevModel>(int, size_t);
}  // namespace dmx
