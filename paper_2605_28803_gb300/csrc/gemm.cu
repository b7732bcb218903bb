// Dispatch of the W4A4 GEMM (the kernel template lives in gemm_kernel.cuh): tile shapes and
// orientations for each launch, and the device error word of the kernels instantiated here.
#include "gemm_kernel.cuh"

namespace qvla {
namespace {

// Per-group step scales: int4 operand bytes, 128-wide tiles at most (the running sum takes a
// third TMEM region).
template <typename OutT>
cudaError_t launch_grouped(const GemmArgs& a) {
  if (a.gated || a.x_bytes != 1) return cudaErrorInvalidValue;
  if (a.M > 128) return launch_cfg<128, false, false, 1, OutT, true>(a);
  const int mpad = (a.M + 15) / 16 * 16;
  if (mpad <= 16) return launch_cfg<16, true, false, 1, OutT, true>(a);
  if (mpad <= 32) return launch_cfg<32, true, false, 1, OutT, true>(a);
  if (mpad <= 64) return launch_cfg<64, true, false, 1, OutT, true>(a);
  return launch_cfg<128, true, false, 1, OutT, true>(a);
}

// Token-major tile shapes and their estimated launch times (ns): a fixed cost plus, per wave of
// persistent CTAs (or CTA pairs), a per-tile cost and a cost per k-block, fitted to GB300
// measurements (M 256-8192, K 1024-16384; pairs only from K = 1024): single CTAs with 128- / 256-wide tiles 2300 + waves x
// (2000 + 344 / k-block) and 2000 + waves x (2500 + 560 / k-block); CTA pairs (256 tokens over two
// SMs, half the weight rows staged per SM) 3900 + waves x (1000 + 351 / k-block) and 3800 + waves
// x (2900 + 375 / k-block).  A pair wave holds half as many tiles, each of twice the tokens.
enum class TileShape { kSingle128, kSingle256, kPair128, kPair256 };

TileShape token_major_shape(const GemmArgs& a, long* estimate = nullptr) {
  const long nkb = a.K / kBK, sms = a.num_sms, npairs = a.num_sms / 2;
  const long t1 = (a.M + kBM - 1) / kBM, t2 = (a.M + 2 * kBM - 1) / (2 * kBM);
  const long n128 = a.gated ? 0 : (a.N + 127) / 128, n256 = (a.N + 255) / 256;
  auto est = [&](long tiles, long units, long fixed, long per_tile, long per_kb) {
    return fixed + (tiles + units - 1) / units * (per_tile + nkb * per_kb);
  };
  TileShape best = TileShape::kSingle256;
  long t = est(t1 * n256, sms, 2000, 2500, 560);
  auto consider = [&](TileShape s, long v) {
    if (v < t) {
      t = v;
      best = s;
    }
  };
  if (n128) consider(TileShape::kSingle128, est(t1 * n128, sms, 2300, 2000, 344));
  // pairs need a few k-blocks per tile to hide their larger per-tile hand-over (measured at
  // K = 256: 12% slower than single CTAs where this estimate favoured the pair)
  if (a.M > kBM && npairs > 0 && nkb >= 8) {
    consider(TileShape::kPair256, est(t2 * n256, npairs, 3800, 2900, 375));
    if (n128) consider(TileShape::kPair128, est(t2 * n128, npairs, 3900, 1000, 351));
  }
  if (estimate) *estimate = t;
  return best;
}

// Whether the kernel with the weights in TMEM takes the launch, with its plan.  From K = 768 it was faster than the
// token-major kernel at every shape measured (M 129-8192 and gated M 5-128, N 16-32768: 1.04 to 2.8 times); below, the
// estimates decide.  Up to 128 tokens a layer that is not gated keeps the weight-major kernel: alone the other is faster
// from K N = 2^21 or so, but between the small kernels of a chain it is not (the action head's step at 50 tokens: 240
// against 221 us), as its pairs fill the SMs' shared memory and TMEM and so start late.  Packed 4-bit codes go by the estimates
// at every K, the token-major one an eighth up, as it was fitted to operand bytes (2328 x 3200 -> 1536: 19.0 us token-major
// and 20.2 here; 400 x 2048 -> 8192 14.2 and 14.7; 1000 x 1024 -> 16384 30.2 and 24.7).
bool take_tmem(const GemmArgs& a, int* bn, int* parts) {
  if (a.num_sms < 2 || (!a.gated && a.M <= 128)) return false;
  const long t = gemm_tmem_plan(a, bn, parts);
  if (a.K >= 768 && a.x_bytes != 0) return true;
  long old = 0;
  token_major_shape(a, &old);
  if (a.x_bytes == 0) old += old / 8;
  if (a.gated && old < 6900) old = 6900;  // a gated tile's epilogue outlasts a few k-blocks
  return t < old;
}

// 8-bit activation planes on single CTAs: whether 128-wide tiles beat 256-wide ones, by waves x tile width (a gated layer's
// gate and up rows share a 256-row tile).
bool a8_narrow(const GemmArgs& a) {
  const long tm = (a.M + kBM - 1) / kBM;
  const long w256 = (tm * ((a.N + 255) / 256) + a.num_sms - 1) / a.num_sms;
  const long w128 = (tm * ((a.N + 127) / 128) + a.num_sms - 1) / a.num_sms;
  return !a.gated && w128 * 128 < w256 * 256;
}

template <int kX, typename OutT>
cudaError_t launch_out(const GemmArgs& a) {
  int bn = 0, parts = 1;
  if (take_tmem(a, &bn, &parts)) return launch_gemm_tmem(a, bn, parts);
  if (a.gated || a.M > 128) {
    if constexpr (kX == 2) {
      if (a.gated) return launch_cfg<256, false, true, kX, OutT>(a);
      return a8_narrow(a) ? launch_cfg<128, false, false, kX, OutT>(a) : launch_cfg<256, false, false, kX, OutT>(a);
    } else {
      // gated layers always take 256-wide tiles: a tile's gate and up rows meet in one epilogue.  Operand bytes come here
      // below K = 768 only, where no pairs are planned.
      const TileShape shape = token_major_shape(a);
      if constexpr (kX == 0) {
        if (shape == TileShape::kPair256)
          return a.gated ? launch_cfg<256, false, true, kX, OutT, false, true>(a)
                         : launch_cfg<256, false, false, kX, OutT, false, true>(a);
        if (shape == TileShape::kPair128) return launch_cfg<128, false, false, kX, OutT, false, true>(a);
      }
      if (shape == TileShape::kSingle128) return launch_cfg<128, false, false, kX, OutT>(a);
      return a.gated ? launch_cfg<256, false, true, kX, OutT>(a) : launch_cfg<256, false, false, kX, OutT>(a);
    }
  }
  const int mpad = (a.M + 15) / 16 * 16;
  if (mpad <= 16) return launch_cfg<16, true, false, kX, OutT>(a);
  if (mpad <= 32) return launch_cfg<32, true, false, kX, OutT>(a);
  if (mpad <= 64) return launch_cfg<64, true, false, kX, OutT>(a);
  return launch_cfg<128, true, false, kX, OutT>(a);
}

}  // namespace

int gemm_plan(const GemmArgs& a, int* parts) {
  int bn = 0;
  *parts = 1;
  if (take_tmem(a, &bn, parts)) return 3 + bn / 32;
  *parts = 1;
  if (a.x_bytes == 2) return static_cast<int>(a8_narrow(a) ? TileShape::kSingle128 : TileShape::kSingle256);
  return static_cast<int>(token_major_shape(a));
}

cudaError_t launch_gemm_w4a4(const GemmArgs& a) {
  if (a.M == 0) return cudaSuccess;
  {  // one to four tokens: the weight stream decides, so the CUDA-core GEMV takes it
    bool launched = false;
    const cudaError_t e = launch_gemv_w4a4(a, &launched);
    if (e != cudaSuccess || launched) return e;
  }
  if (a.gscale) return a.ydt == 0 ? launch_grouped<__half>(a) : launch_grouped<__nv_bfloat16>(a);
  if (a.x_bytes == 2) return a.ydt == 0 ? launch_out<2, __half>(a) : launch_out<2, __nv_bfloat16>(a);
  if (a.x_bytes == 1) return a.ydt == 0 ? launch_out<1, __half>(a) : launch_out<1, __nv_bfloat16>(a);
  return a.ydt == 0 ? launch_out<0, __half>(a) : launch_out<0, __nv_bfloat16>(a);
}

cudaError_t set_debug_hooks_gemm(unsigned long long wait_limit_ns, int hold_loads) {
  return set_debug_hooks(wait_limit_ns, hold_loads);
}

cudaError_t read_and_clear_error_word(unsigned int* out, cudaStream_t stream) {
  cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyFromSymbol(out, g_error_word, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  const unsigned int zero = 0;
  return cudaMemcpyToSymbol(g_error_word, &zero, sizeof(unsigned int));
}

}  // namespace qvla
