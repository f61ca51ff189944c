// Stencil kernels with bf16 spinor storage, two threads per site.
#include "hop_pair.cuh"

namespace oq {
cudaError_t launch_hop_pair_bf16(const HopLaunch& L, const HopArgs& a, cudaStream_t s) {
  return pair_dispatch<P_BF16>(L, a, s);
}
}  // namespace oq
