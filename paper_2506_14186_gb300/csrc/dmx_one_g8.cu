// Kernels of one-body models (OneBody), 8 lanes per environment: the fused
// rollout, the reverse adjoint without and with parameter gradients.
#include "dmx_adjoint_rev.cuh"
#include "dmx_kernels.cuh"

namespace dmx {
template cudaError_t launch_persistent_g<8, OneBody>(const RolloutParams&, int, int, size_t, cudaStream_t);
template int occupancy_g<8, OneBody>(int, size_t);
template cudaError_t launch_adjoint_rev_g<8, false, OneBody>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<8, false, OneBody>(int, size_t);
template cudaError_t launch_adjoint_rev_g<8, true, OneBody>(const AdjParams&, int, int, size_t, cudaStream_t);
template int occupancy_adjoint_rev_g<8, true, OneBody>(int, size_t);
}  // namespace dmx
