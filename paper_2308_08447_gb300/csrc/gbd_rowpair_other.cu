// The paired x-row kernels (gbd_rowpair.cuh) of the other epilogues: H_eff, dm/dt, general RK stages.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_other(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  auto f = [&](auto l) { pair_launch<decltype(l)::value, 2>(a, tw, st); };
  return pair_switch<0>(Lx, f) || pair_switch<1>(Lx, f);
}
}  // namespace gbd
