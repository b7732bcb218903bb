// Rotate + quantise kernels with 8-bit codes for bf16 activations (the template lives in rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_a8_bf16(const RotQuantArgs& a) {
  return a.out_mode == 2 ? rq::launch_wide<__nv_bfloat16, 2>(a) : rq::launch_wide<__nv_bfloat16, 3>(a);
}
}  // namespace qvla
