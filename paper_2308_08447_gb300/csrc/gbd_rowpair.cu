// The paired x-row kernels (gbd_rowpair.cuh) of the RK4 stages.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_rk(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  return pair_switch<0>(Lx, [&](auto l) { pair_launch<decltype(l)::value, 0>(a, tw, st); });
}
bool pair_dispatch_epi(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  if (!a) return pair_dispatch_rk(Lx, a, tw, st) || pair_dispatch_rk_mixed(Lx, a, tw, st) ? pair_dispatch_other(Lx, a, tw, st) : false;
  if (a->mode >= ROW_RK1 && a->mode <= ROW_RK4) return pair_dispatch_rk(Lx, a, tw, st) || pair_dispatch_rk_mixed(Lx, a, tw, st);
  return pair_dispatch_other(Lx, a, tw, st);
}
}  // namespace gbd
