// Dispatch of the rotate + quantise kernels by activation dtype.
#include "kernels.h"

namespace qvla {

cudaError_t launch_rotate_quant_f16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_bf16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_f32(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_wide_f16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_wide_bf16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_wide_f32(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_a8_f16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_a8_bf16(const RotQuantArgs& a);
cudaError_t launch_rotate_quant_a8_f32(const RotQuantArgs& a);

// The kernel with 32 channels per thread (rotate_quant_wide.cuh): 4-bit codes with one scale per row (per token or per
// step), or per step and group of up to 1024 channels, whose 32 threads sum their codes within a warp.  K is a multiple of
// 128 and of the block, which is all that its groups of threads need.
static bool rotate_quant_wide_takes(const RotQuantArgs& a) {
  const bool rows = a.gshift >= 30 && a.xgsum == nullptr, groups = a.mode == 1 && a.gshift <= 10;
  return (a.mode == 0 || a.mode == 1) && (a.out_mode == 0 || a.out_mode == 1) && (rows || groups) && a.log_b >= 0 && a.log_b <= 12;
}

bool rotate_quant_supported(int log_b) { return log_b >= 0 && log_b <= 12; }

cudaError_t launch_rotate_quant(const RotQuantArgs& a) {
  {  // operand bytes of 16-bit activations, one scale per row: one CTA per 2048-channel pass
    bool launched = false;
    const cudaError_t e = launch_rotate_quant_pass(a, &launched);
    if (e != cudaSuccess || launched) return e;
  }
  if (a.out_mode >= 2) {  // 8-bit codes, one scale per row
    switch (a.xdt) {
      case 0: return launch_rotate_quant_a8_f16(a);
      case 1: return launch_rotate_quant_a8_bf16(a);
      case 2: return launch_rotate_quant_a8_f32(a);
      default: return cudaErrorInvalidValue;
    }
  }
  if (rotate_quant_wide_takes(a)) {
    switch (a.xdt) {
      case 0: return launch_rotate_quant_wide_f16(a);
      case 1: return launch_rotate_quant_wide_bf16(a);
      case 2: return launch_rotate_quant_wide_f32(a);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (a.xdt) {
    case 0: return launch_rotate_quant_f16(a);
    case 1: return launch_rotate_quant_bf16(a);
    case 2: return launch_rotate_quant_f32(a);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qvla
