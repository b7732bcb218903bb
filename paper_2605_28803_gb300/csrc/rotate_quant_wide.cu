// Rotate + quantise kernels with 32 channels per thread, 4-bit codes (the template lives in rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_wide_f16(const RotQuantArgs& a) {
  return a.out_mode == 0 ? rq::launch_wide<__half, 0>(a) : rq::launch_wide<__half, 1>(a);
}
cudaError_t launch_rotate_quant_wide_bf16(const RotQuantArgs& a) {
  return a.out_mode == 0 ? rq::launch_wide<__nv_bfloat16, 0>(a) : rq::launch_wide<__nv_bfloat16, 1>(a);
}
}  // namespace qvla
