// row_kernel for the transform lengths Lx = 3 * 2^k and 5 * 2^k from 320 (FP32; gbd_fft.cuh), one tile
// shape each: the launches whose blocks make one wave over the GPU, where its four to six times the
// threads per row outrun the paired rows (take_pair in gbd_row.cu).
#include "gbd_row.cuh"

namespace gbd {

bool row_dispatch_mixed(int Lx, const RowArgs* a, const float2* tw, cudaStream_t st) {
  switch (Lx) {
#define GBD_MIXED_ROW(LX)                            \
  case LX:                                           \
    row_launch_t<LX, row_rb(LX, 0), 0>(a, tw, st);   \
    return true;
    GBD_MIXED_ROW(320)
    GBD_MIXED_ROW(384)
    GBD_MIXED_ROW(640)
    GBD_MIXED_ROW(768)
    GBD_MIXED_ROW(1280)
    GBD_MIXED_ROW(1536)
    GBD_MIXED_ROW(2560)
    GBD_MIXED_ROW(3072)
#undef GBD_MIXED_ROW
    default: return false;
  }
}

}  // namespace gbd
