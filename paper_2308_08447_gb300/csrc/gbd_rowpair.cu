// The paired x-row kernels (gbd_rowpair.cuh) with an epilogue.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_epi(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  return pair_switch<0>(Lx, [&](auto l) { pair_launch<decltype(l)::value, 0>(a, tw, st); });
}
}  // namespace gbd
