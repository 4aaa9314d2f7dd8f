// The paired x-row kernels (gbd_rowpair.cuh) of the RK4 stages, lengths 3 * 2^k and 5 * 2^k.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_rk_mixed(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  return pair_switch<1>(Lx, [&](auto l) { pair_launch<decltype(l)::value, 0>(a, tw, st); });
}
}  // namespace gbd
