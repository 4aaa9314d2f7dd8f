// The paired x-row kernels (gbd_rowpair.cuh) of the transform-only launches.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_io(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  auto f = [&](auto l) { pair_launch<decltype(l)::value, 1>(a, tw, st); };
  return pair_switch<0>(Lx, f) || pair_switch<1>(Lx, f);
}
}  // namespace gbd
