// The paired x-row kernels (gbd_rowpair.cuh) with an epilogue, lengths 3 * 2^k and 5 * 2^k.
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_epi_mixed(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  return pair_switch<1>(Lx, [&](auto l) { pair_launch<decltype(l)::value, 0>(a, tw, st); });
}
}  // namespace gbd
