// Kernels of models without geom pairs (PlaneOnly), 32 lanes per environment:
// the fused rollout and the reverse adjoint.
#include "dmx_adjoint_rev.cuh"
#include "dmx_kernels.cuh"

namespace dmx {
template cudaError_t launch_persistent_g<32, PlaneOnly>(const RolloutParams&, int, int, size_t, cudaStream_t);
template int occupancy_g<32, PlaneOnly>(int, size_t);
template cudaError_t launch_adjoint_rev_g<32, false, PlaneOnly>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<32, false, PlaneOnly>(int, size_t);
}  // namespace dmx
