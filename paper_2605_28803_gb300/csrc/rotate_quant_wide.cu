// Rotate + quantise kernels with 32 channels per thread (the template lives in rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_wide_f16(const RotQuantArgs& a) { return rq::launch_wide<__half>(a); }
cudaError_t launch_rotate_quant_wide_bf16(const RotQuantArgs& a) { return rq::launch_wide<__nv_bfloat16>(a); }
}  // namespace qvla
