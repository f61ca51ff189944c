// Stencil kernels with f16 spinor storage, two threads per site.
#include "hop_pair.cuh"

namespace oq {
cudaError_t launch_hop_pair_f16(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  return pair_dispatch<P_F16>(L, a, s);
}
}  // namespace oq
