// The paired x-row kernels (gbd_rowpair.cuh) of the transform-only launches (powers of two: below 1024,
// take_pair in gbd_row.cu).
#include "gbd_rowpair.cuh"

namespace gbd {
bool pair_dispatch_io(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  auto f = [&](auto l) {
    constexpr int L = decltype(l)::value;
    if constexpr (mixed_len(L) || L < 1024) pair_launch<L, 1>(a, tw, st);
  };
  return pair_switch<0>(Lx, f) || pair_switch<1>(Lx, f);
}
}  // namespace gbd
