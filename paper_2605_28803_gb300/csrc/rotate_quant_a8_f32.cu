// Rotate + quantise kernels with 8-bit codes for f32 activations (the template lives in rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_a8_f32(const RotQuantArgs& a) {
  return a.out_mode == 2 ? rq::launch_wide<float, 2>(a) : rq::launch_wide<float, 3>(a);
}
}  // namespace qvla
