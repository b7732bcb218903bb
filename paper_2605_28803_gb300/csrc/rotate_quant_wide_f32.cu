// Rotate + quantise kernels with 32 channels per thread for f32 activations, 4-bit codes (the template lives in
// rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_wide_f32(const RotQuantArgs& a) {
  return a.out_mode == 0 ? rq::launch_wide<float, 0>(a) : rq::launch_wide<float, 1>(a);
}
}  // namespace qvla
