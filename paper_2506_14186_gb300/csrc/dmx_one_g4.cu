// Kernels of one-body models (OneBody), 4 lanes per environment: the fused
// rollout.
#include "dmx_adjoint_rev.cuh"
#include "dmx_kernels.cuh"

namespace dmx {
template cudaError_t launch_persistent_g<4, OneBody>(const RolloutParams&, int, int, size_t, cudaStream_t);
template int occupancy_g<4, OneBody>(int, size_t);
}  // namespace dmx
