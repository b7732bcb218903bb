// Rotate + quantise kernels with 32 channels per thread for f32 activations (the template lives in rotate_quant_wide.cuh).
#include "rotate_quant_wide.cuh"

namespace qvla {
cudaError_t launch_rotate_quant_wide_f32(const RotQuantArgs& a) { return rq::launch_wide<float>(a); }
}  // namespace qvla
