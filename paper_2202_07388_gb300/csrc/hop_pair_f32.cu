// Stencil kernels with f32 spinor storage, two threads per site.
#include "hop_pair.cuh"

namespace oq {
cudaError_t launch_hop_pair_f32(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  return pair_dispatch<P_F32>(L, a, s);
}
}  // namespace oq
