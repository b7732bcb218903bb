// Fused online rotation + symmetric 4-bit or 8-bit activation quantisation (Sec. 4.1 Eq. 3-5, Sec. 4.2 Eq. 5-6) for batches of
// rows: 32 channels per thread, 4-bit codes by packed E4M3 conversion, 8-bit codes by magic-number rounding.
//
// It does what rotate_quant.cuh's kernel does, bit for bit, with fewer instructions
// per channel and twice the warps in flight:
//   * a thread holds 32 channels instead of 64: 64 registers, 32 warps per SM.  (19 of the 312 instances, all with a scale per
//     step, spill 4 to 24 bytes a thread there, most with blocks of 512: -Xptxas -v);
//   * the butterflies run in three phases, index bits 0-4 on 32 consecutive channels, 5-7 (5-6 among 4 threads for blocks of
//     64 and 128, whose rows need not be whole 256-channel groups), and 8-10 (8-11 for blocks of 4096, on half quads), with a transpose through shared memory between phases whose stores and loads both move 16
//     bytes (4 channels, a quad) per thread.  A quad is the channels whose codes fill one 32-bit word of the output, so after the last phase every code leaves in a
//     4-byte store, 128 contiguous bytes per warp (the 64-channel layout ends in 1-byte stores at b = 2048).  The stage
//     order and every rounding are the other kernel's;
//   * a code q is the E4M3 byte of (q + 8) 2^-9, so one conversion instruction rounds two values to operand bytes.  It is
//     done twice, with the value moved up and down by 2^-16 of a step: equal bytes mean that no value is near a rounding
//     tie, where the other kernel's fast path gives the same code; otherwise (and for a byte that is no code: a NaN, or a
//     clamp that an overflowing reciprocal asks for) the quads take that kernel's arithmetic, exact decision included.
//     Rows whose reciprocal scale is so small or large that its product with 2^-9 could lose bits take it throughout.
//
// Measured back to back in a graph, 64-channel kernel before and this one, us: 816 x 2048 bf16 5.9 and 4.8; 816 x 16384
// 23.0 and 18.0; 3200 x 16384 f16 72.0 and 58.4 (2.7 TB/s of x and codes); 8192 x 2048 22.7 and 19.3; 201 x 2304 with
// blocks of 256 3.9 and 2.8; f32 777 x 4096 9.9 and 9.7; blocks of 128: 3325 x 10112 47.3 and 32.0, 7761 x 2688 29.3 and 20.6,
// 8192 x 384 8.6 and 5.2; with a scale per 128-channel group the linear 50 x 1024 -> 4096 8.0 and 7.0, 5954 x 14080 -> 288
// 233 and 223.  8-bit codes: the gated linear 816 x 2048 -> 2 x 16384 73.5 and 70.7, one row of 1536 -> 5168 8.5 and 7.0.  About 21 instructions a channel at 55% of the issue slots; neither
// the transposes, the butterflies nor the conversions alone bound it (leaving one of them out saves 6 to 16%).  Staying
// CTAs fed by TMA one group ahead were slower (73 us at 3200 x 16384): with an extra barrier a group, two CTAs an SM overlap
// less than fresh ones.  A few rows are spread one to a CTA: 50 x 1024 2.1 us against 2.8 with eight rows a CTA; with blocks
// of 4096 at 50 x 4096 (128 channels a thread in the other kernel) the action head's step went from 208 to 188 us.
#pragma once

#include "ptx.cuh"
#include "rotate_quant.cuh"

namespace qvla {
namespace rq {

constexpr int kWideThreads = 512;  // most threads of a CTA (K = 16384: one row)
constexpr int kWideRows = 64;      // most rows of a CTA

// Four values as E4M3 bytes (round to nearest even), in order.
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  uint16_t lo, hi;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(b), "f"(a));  // the second operand is the low byte
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(d), "f"(c));
  return static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
}

__device__ __forceinline__ void sts128(uint32_t addr, float2 a, float2 b) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y) : "memory");
}
__device__ __forceinline__ void lds64(uint32_t addr, float2& a) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(a.x), "=f"(a.y) : "r"(addr) : "memory");
}
__device__ __forceinline__ void lds128(uint32_t addr, float2& a, float2& b) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a.x), "=f"(a.y), "=f"(b.x), "=f"(b.y) : "r"(addr) : "memory");
}

// The threads of a Hadamard block meet between the second and the third phase: part of a warp, or two or four warps.
template <int kLogB>
__device__ __forceinline__ void block_sync() {
  if constexpr (kLogB <= 10) {
    __syncwarp();
  } else {  // 64 or 128 threads
    asm volatile("bar.sync %0, %1;" ::"r"(1 + static_cast<int>(threadIdx.x >> (kLogB - 5))), "n"(1 << (kLogB - 5)) : "memory");
  }
}

// The codes of four values (operand bytes q + 8) by the other kernel's arithmetic.
static __device__ __noinline__ uint32_t codes4_exact(float4 y, float inv_sqrt_b, float delta, float cr, bool step, bool all) {
  const float v[4] = {y.x, y.y, y.z, y.w};
  float u[4];
  float dev = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float t = __fmul_rn(v[i], cr);
    if (step) t = fminf(fmaxf(t, -7.0f), 7.0f);
    u[i] = __fadd_rn(t, kMagic);
    dev = fmaxf(dev, fabsf(__fmaf_rn(__fadd_rn(u[i], -kMagic), -1.0f, t)));
  }
  if (dev >= kTieBand || all) {
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = exact_code(v[i], inv_sqrt_b, delta, cr, 7.0f, kTieBand);
  }
  return (low_bytes(u[0], u[1], u[2], u[3]) & 0x0F0F0F0Fu) ^ 0x08080808u;
}

// kOut, the output: 0 packed nibbles [M][K/2], 1 operand bytes [M][K]; 8-bit codes: 2 int8 rows [M][K], 3 the GEMM's two operand
// planes [M][2 K].  In 0 and 2 a quad is 4 consecutive channels; in 1 and 3, where each group of 8 is stored k0 k2 k4 k6 k1 k3
// k5 k7, its even or its odd ones.  8-bit codes are rounded by the other kernel's arithmetic (no E4M3 byte holds them).
template <typename T, int kLogB, bool kStep, int kOut>
__global__ void __launch_bounds__(kWideThreads, 2) rotate_quant_wide_kernel(const T* __restrict__ x, int M, int K, float inv_sqrt_b,
                                                                            const float* __restrict__ step_scale,
                                                                            uint8_t* __restrict__ xq, float* __restrict__ xscale,
                                                                            int32_t* __restrict__ xsum, int gshift,
                                                                            int32_t* __restrict__ xgsum,
                                                                            int32_t* __restrict__ zero, int zero_n) {
  constexpr int kA = kLogB < 5 ? kLogB : 5;                        // index bits of the first phase
  constexpr int kRB = kLogB <= 5 ? 0 : kLogB < 8 ? kLogB - 5 : 3;  // of the second: 5 .. 5 + kRB - 1
  constexpr int kRC = kLogB <= 8 ? 0 : kLogB - 8;                  // of the third: 8 .. 8 + kRC - 1
  // blocks of 64 and 128: the second phase trades among 4 threads, so that a row needs whole 128-channel groups only
  constexpr bool kFour = kRB == 1 || kRB == 2;
  constexpr bool kHalf = kRC == 4;  // after the third phase a thread holds half quads (two channels) of 16 lines
  static_assert(kLogB <= 12, "Hadamard blocks up to 4096");
  constexpr bool kPacked = kOut == 0, kNatural = kOut == 0 || kOut == 2, kA8 = kOut >= 2;
  constexpr float kQ = kA8 ? 127.0f : 7.0f;
  extern __shared__ __align__(128) uint8_t wide_smem[];  // one line of 8 quads (128 bytes) per thread
  __shared__ unsigned int s_max[kWideRows], s_sum[kWideRows];

  const int tpr = K >> 5, rpc = blockDim.x / tpr;
  const int tid = threadIdx.x;
  const int rloc = tid / tpr, j = tid - rloc * tpr;
  const int m = blockIdx.x * rpc + rloc;
  const bool active = rloc < rpc && m < M;
  const bool one_warp = tpr == 32;  // a row is a warp: no shared reduction
  // a warp within one row reduces as a warp; else its groups of 4 threads (K is a multiple of 128), if whole
  const bool row_warp = __shfl_sync(0xffffffffu, rloc, 0) == __shfl_sync(0xffffffffu, rloc, 31);
  if (tid < kWideRows) {
    s_max[tid] = 0u;
    s_sum[tid] = 0u;
  }
  griddep_wait();  // x comes from the previous kernel, which may still read xq / xscale / xsum
  griddep_launch_dependents();
  if (zero != nullptr && blockIdx.x == 0)  // the next GEMM's work-unit counters (its previous use is over)
    for (int i = tid; i < zero_n; i += blockDim.x) zero[i] = 0;
  float2 v[16];
  if (active) {
    const T* src = x + static_cast<size_t>(m) * K + static_cast<size_t>(j) * 32;
#pragma unroll
    for (int c = 0; c < 32 / Loader<T>::kPer16B; ++c) Loader<T>::load(src + c * Loader<T>::kPer16B, v + c * (Loader<T>::kPer16B / 2));
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = make_float2(0.0f, 0.0f);
  }
  if (!one_warp) __syncthreads();  // the reduction slots are cleared before any thread adds to them
  // phase 1, leaving v as quads: quad q of the 32-channel line in v[2 q], v[2 q + 1]
  if constexpr (kNatural) {
    fwht_regs<16, 0, kA>(v);
  } else {
    // quad i0 + 2 g: the even (i0 = 0) or odd channels of group g, paired like that before the butterflies (the pair's own
    // lane is then index bit 1, bit 0 lies two registers apart), so that no value moves between them
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float2 a = v[4 * g], b = v[4 * g + 1], c = v[4 * g + 2], d = v[4 * g + 3];
      v[4 * g] = make_float2(a.x, b.x);
      v[4 * g + 1] = make_float2(c.x, d.x);
      v[4 * g + 2] = make_float2(a.y, b.y);
      v[4 * g + 3] = make_float2(c.y, d.y);
    }
    if constexpr (kA > 0) {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if ((i & 2) == 0) bfly2(v[i], v[i + 2]);
    }
    if constexpr (kA > 1) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float a = v[i].x, c = v[i].y;
        v[i] = make_float2(a + c, a - c);
      }
    }
#pragma unroll
    for (int bit = 2; bit < kA; ++bit) {  // bits 2, 3, 4: one, four, eight registers apart
      const int h = bit == 2 ? 1 : 1 << (bit - 1);
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if ((i & h) == 0) bfly2(v[i], v[i + h]);
    }
  }
  const int q = j & 7;  // after a transpose: this thread's quad of every line it holds
  // quad i of line l lies at piece i ^ (l % 8) of the line's 128 bytes: stores and loads of 8 threads meet 8 pieces
  const uint32_t lines = smem_u32(wide_smem);
  const uint32_t own = lines + static_cast<uint32_t>(tid * 128 + q * 16);
  if constexpr (kFour) {
    // phase 2: thread p of the 4 of a 128-channel group takes quads 2 p and 2 p + 1 of its lines.  Quad i of line l at piece
    // i ^ s(l), s = 0 2 4 6 1 3 5 7 over 8 lines: the even pieces two groups read at a time fall on all eight
    const int g = (tid >> 2) & 1, p = tid & 3;
    const uint32_t line = lines + static_cast<uint32_t>(tid * 128 + (2 * p + g) * 16);
#pragma unroll
    for (int i = 0; i < 8; ++i) sts128(line ^ static_cast<uint32_t>(i * 16), v[2 * i], v[2 * i + 1]);
    __syncwarp();
    const uint32_t grp = lines + static_cast<uint32_t>((tid & ~3) * 128 + ((2 * p) ^ g) * 16);
#pragma unroll
    for (int i = 0; i < 8; ++i)  // i = 2 l + e
      lds128((grp ^ static_cast<uint32_t>(i * 16)) + (i >> 1) * 128, v[2 * i], v[2 * i + 1]);
    fwht_regs<16, 3, 3 + kRB>(v);
  } else if constexpr (kRB > 0) {
    // phase 2: the 8 threads of a 256-channel group trade quads for lines; line l of the group at thread l's place
#pragma unroll
    for (int i = 0; i < 8; ++i) sts128(own ^ static_cast<uint32_t>(i * 16), v[2 * i], v[2 * i + 1]);
    __syncwarp();
    const uint32_t grp = lines + static_cast<uint32_t>((tid & ~7) * 128 + q * 16);
#pragma unroll
    for (int l = 0; l < 8; ++l) lds128((grp ^ static_cast<uint32_t>(l * 16)) + l * 128, v[2 * l], v[2 * l + 1]);
    fwht_regs<16, 2, 2 + kRB>(v);
  }
  if constexpr (kRC > 0) {
    // phase 3: the 8 * 2^kRC threads (h, q) of a Hadamard block trade the high kRC bits of the line for the group index h
    constexpr int kLb = kHalf ? 0 : 3 - kRC;  // line bits a thread keeps
    __syncwarp();                             // the group has read this thread's lines
#pragma unroll
    for (int l = 0; l < 8; ++l) sts128(own ^ static_cast<uint32_t>(l * 16), v[2 * l], v[2 * l + 1]);
    block_sync<kLogB>();
    constexpr int kGroup = 8 << kRC;
    if constexpr (kHalf) {  // thread (l, q, e) of the block: half e of quad q of line l of all 16 groups
      const int l = (j >> 4) & 7, qq = (j >> 1) & 7;
      const uint32_t blk = lines + static_cast<uint32_t>((tid & ~(kGroup - 1)) * 128 + qq * 128 + ((l ^ qq) << 4) + (j & 1) * 8);
#pragma unroll
      for (int h = 0; h < 16; ++h) lds64(blk + h * 1024, v[h]);
      fwht_regs<16, 1, 5>(v);
    } else {
      const int la = (j >> 3) & ((1 << kRC) - 1);
      const uint32_t blk = (lines + static_cast<uint32_t>((tid & ~(kGroup - 1)) * 128 + q * 144)) ^ static_cast<uint32_t>(la << (kLb + 4));
#pragma unroll
      for (int i = 0; i < 8; ++i)
        lds128((blk ^ static_cast<uint32_t>((i & ((1 << kLb) - 1)) * 16)) + (i >> kLb) * 1024, v[2 * i], v[2 * i + 1]);
      fwht_regs<16, kHalf ? 5 : 5 - kRC, 5>(v);
    }
  }

  // ---- scale ----
  float delta;
  if constexpr (kStep) {
    // (a scale group holds whole Hadamard blocks of at most 32 threads: this thread's channels stay in one)
    delta = __ldg(step_scale + (gshift >= 30 ? 0 : (j * 32) >> gshift));
  } else {
    float w = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) w = max_nan(w, max_nan(fabsf(v[i].x), fabsf(v[i].y)));
    unsigned int wm = __float_as_uint(w);  // non-negative floats order as their bit patterns, NaN above infinity
    if (row_warp) {
      wm = __reduce_max_sync(0xffffffffu, wm);
      if (!one_warp && (tid & 31) == 0 && rloc < rpc) atomicMax(&s_max[rloc], wm);
    } else {
      wm = max(wm, __shfl_xor_sync(0xffffffffu, wm, 1));
      wm = max(wm, __shfl_xor_sync(0xffffffffu, wm, 2));
      if ((tid & 3) == 0 && rloc < rpc) atomicMax(&s_max[rloc], wm);
    }
    if (!one_warp) {
      __syncthreads();
      wm = s_max[rloc < rpc ? rloc : 0];
    }
    // max |Z| of the normalised rotation: rounding is monotone, so round(max * c) = max round(y * c)
    delta = __fdiv_rn(__uint_as_float(wm) * inv_sqrt_b, kQ);
  }
  if (active && j == 0) xscale[m] = delta;

  // ---- codes: quad i of this thread as operand bytes q + 8 (8-bit codes: as they are) ----
  const bool zero_scale = !(delta > 0.0f);
  const float rcp = zero_scale ? 0.0f : __frcp_rn(delta);
  const bool tiny_scale = !zero_scale && isinf(rcp);  // 1 / delta overflows: plain division
  const float cr = inv_sqrt_b * rcp;                  // y * cr ~ z / delta (0 when delta = 0: codes 0)
  // the scaled product below could lose bits (a zero cannot: a row of zeros, such as padding, stays on the fast path, where
  // its codes are 0 exactly; sent the other way, 3200 x 16384 f16 zeros took 76 us)
  const bool plain = cr != 0.0f && !(cr >= 1e-30f && cr <= 1e30f);
  const float2 cr9 = make_float2(cr * 0.001953125f, cr * 0.001953125f);
  // (8 +- 2^-16) 2^-9
  const float2 up = make_float2(0.0156250298023223876953125f, 0.0156250298023223876953125f);
  const float2 dn = make_float2(0.0156249701976776123046875f, 0.0156249701976776123046875f);
  uint32_t code[8];
  uint32_t sum_acc = 0;
  if constexpr (kA8) {
    const float2 cr2 = make_float2(cr, cr), magic2 = make_float2(kMagic, kMagic);
    const float2 nmagic2 = make_float2(-kMagic, -kMagic), neg2 = make_float2(-1.0f, -1.0f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float2 u[2];
      float dev = 0.0f;  // the largest distance |t - round(t)| of the quad
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float2 t = __fmul2_rn(v[2 * i + k], cr2);
        if constexpr (kStep) t = make_float2(fminf(fmaxf(t.x, -kQ), kQ), fminf(fmaxf(t.y, -kQ), kQ));
        u[k] = __fadd2_rn(t, magic2);
        const float2 d = __ffma2_rn(__fadd2_rn(u[k], nmagic2), neg2, t);
        dev = fmaxf(dev, fmaxf(fabsf(d.x), fabsf(d.y)));
      }
      if (dev >= kTieBand8 || tiny_scale) {  // rare: decide these values exactly
#pragma unroll
        for (int k = 0; k < 2; ++k)
          u[k] = make_float2(exact_code(v[2 * i + k].x, inv_sqrt_b, delta, cr, kQ, kTieBand8),
                             exact_code(v[2 * i + k].y, inv_sqrt_b, delta, cr, kQ, kTieBand8));
      }
      code[i] = low_bytes(u[0].x, u[0].y, u[1].x, u[1].y);
      sum_acc = __dp4a(code[i] ^ 0x80808080u, 0x01010101u, sum_acc);
    }
  }
#pragma unroll
  for (int i = 0; i < 8 && !kA8; i += 2) {
    uint32_t odd = 0;  // nonzero: a value near a tie, or no code
#pragma unroll
    for (int k = i; k < i + 2; ++k) {
      float2 a = v[2 * k], b = v[2 * k + 1];
      if constexpr (kStep) {  // t, clamped to [-7, 7]
        const float2 crr = make_float2(cr, cr);
        a = __fmul2_rn(a, crr);
        b = __fmul2_rn(b, crr);
        a = make_float2(fminf(fmaxf(a.x, -7.0f), 7.0f), fminf(fmaxf(a.y, -7.0f), 7.0f));
        b = make_float2(fminf(fmaxf(b.x, -7.0f), 7.0f), fminf(fmaxf(b.y, -7.0f), 7.0f));
      }
      const float2 s2 = kStep ? make_float2(0.001953125f, 0.001953125f) : cr9;
      const float2 ah = __ffma2_rn(a, s2, up), bh = __ffma2_rn(b, s2, up);
      const float2 al = __ffma2_rn(a, s2, dn), bl = __ffma2_rn(b, s2, dn);
      code[k] = e4m3x4(ah.x, ah.y, bh.x, bh.y);
      odd |= (code[k] ^ e4m3x4(al.x, al.y, bl.x, bl.y)) | (code[k] & 0xF0F0F0F0u);
    }
    if (odd != 0u || plain) {
#pragma unroll
      for (int k = i; k < i + 2; ++k)
        code[k] = codes4_exact(make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y), inv_sqrt_b, delta, cr, kStep,
                               tiny_scale);
    }
    sum_acc = __dp4a(code[i], 0x01010101u, sum_acc);
    sum_acc = __dp4a(code[i + 1], 0x01010101u, sum_acc);
  }

  // ---- store ----
  if (active) {
    uint8_t* const dst = xq + static_cast<size_t>(m) * (kPacked ? K / 2 : kOut == 3 ? 2 * K : K);
    // n (1, 2, 4) words of codes at channel o; the planes of a 128-code k-block are 128 bytes each, high nibbles first
    auto put = [&](int o, auto w) {
      using W = decltype(w);
      if constexpr (kOut == 3) {
        W h = w, l = w;
#pragma unroll
        for (int k = 0; k < static_cast<int>(sizeof(W) / 4); ++k) {
          const uint32_t c = reinterpret_cast<const uint32_t*>(&w)[k] ^ 0x80808080u;
          reinterpret_cast<uint32_t*>(&l)[k] = c & 0x0F0F0F0Fu;
          reinterpret_cast<uint32_t*>(&h)[k] = hi_plane_bytes((c >> 4) & 0x0F0F0F0Fu);
        }
        *reinterpret_cast<W*>(dst + o + (o & ~127)) = h;
        *reinterpret_cast<W*>(dst + o + (o & ~127) + 128) = l;
      } else {
        *reinterpret_cast<W*>(dst + o) = w;
      }
    };
    // the two halves of a word 256 channels apart
    auto put_halves = [&](int o, uint32_t w) {
      if constexpr (kOut == 3) {
        const uint32_t c = w ^ 0x80808080u, l = c & 0x0F0F0F0Fu, h = hi_plane_bytes((c >> 4) & 0x0F0F0F0Fu);
        uint8_t* const p = dst + o + (o & ~127);
        *reinterpret_cast<uint16_t*>(p) = static_cast<uint16_t>(h);
        *reinterpret_cast<uint16_t*>(p + 128) = static_cast<uint16_t>(l);
        *reinterpret_cast<uint16_t*>(p + 512) = static_cast<uint16_t>(h >> 16);
        *reinterpret_cast<uint16_t*>(p + 640) = static_cast<uint16_t>(l >> 16);
      } else {
        *reinterpret_cast<uint16_t*>(dst + o) = static_cast<uint16_t>(w);
        *reinterpret_cast<uint16_t*>(dst + o + 256) = static_cast<uint16_t>(w >> 16);
      }
    };
    auto nibbles = [](uint32_t w) -> uint32_t {  // four codes as two packed bytes
      const uint32_t n = w ^ 0x08080808u;
      return __byte_perm(n | (n >> 4), 0u, 0x4420);
    };
    if constexpr (kRB == 0) {  // 32 consecutive channels
      if constexpr (kPacked) {
        *reinterpret_cast<uint4*>(dst + static_cast<size_t>(j) * 16) =
            make_uint4(nibbles(code[0]) | (nibbles(code[1]) << 16), nibbles(code[2]) | (nibbles(code[3]) << 16),
                       nibbles(code[4]) | (nibbles(code[5]) << 16), nibbles(code[6]) | (nibbles(code[7]) << 16));
      } else {
        put(j * 32, make_uint4(code[0], code[1], code[2], code[3]));
        put(j * 32 + 16, make_uint4(code[4], code[5], code[6], code[7]));
      }
    } else if constexpr (kFour) {  // quads 2 p and 2 p + 1 of 4 lines
      const int at = j & ~3, p = j & 3;
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        if constexpr (kPacked) {
          *reinterpret_cast<uint32_t*>(dst + (at + l) * 16 + p * 4) = nibbles(code[2 * l]) | (nibbles(code[2 * l + 1]) << 16);
        } else {
          put((at + l) * 32 + p * 8, make_uint2(code[2 * l], code[2 * l + 1]));
        }
      }
    } else {
      constexpr int kLb = kHalf ? 0 : 3 - kRC;
      const int la = (j >> 3) & ((1 << kRC) - 1);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if constexpr (kHalf) {  // word i: the half quads of groups 2 i and 2 i + 1
          const int at = (j & ~127) + 16 * i + ((j >> 4) & 7), piece = j & 15;  // 8 lines a group
          if constexpr (kPacked) {
            const uint32_t n = nibbles(code[i]);
            dst[at * 16 + piece] = static_cast<uint8_t>(n);
            dst[(at + 8) * 16 + piece] = static_cast<uint8_t>(n >> 8);
          } else {
            put_halves(at * 32 + piece * 2, code[i]);
          }
          continue;
        }
        // the line of quad i: phase 2 leaves line i of the 256-channel group, phase 3 line l of group h of the block
        int line;
        if constexpr (kRC == 0) {
          line = (j & ~7) + i;
        } else {
          line = (j & ~((8 << kRC) - 1)) + (i >> kLb) * 8 + ((la << kLb) | (i & ((1 << kLb) - 1)));
        }
        if constexpr (kPacked) {
          *reinterpret_cast<uint16_t*>(dst + line * 16 + q * 2) = static_cast<uint16_t>(nibbles(code[i]));
        } else {
          put(line * 32 + q * 4, code[i]);
        }
      }
    }
  }
  if (xgsum != nullptr) {  // the code sum of each scale group of the row (at most 32 consecutive lanes)
    int gs = static_cast<int>(sum_acc) - 8 * 32;
    const int tg = 1 << (gshift - 5);
    for (int o = tg >> 1; o > 0; o >>= 1) gs += __shfl_xor_sync(0xffffffffu, gs, o);
    if (active && (j & (tg - 1)) == 0) xgsum[static_cast<size_t>(m) * (K >> gshift) + ((j * 32) >> gshift)] = gs;
  }
  if (xsum != nullptr) {
    unsigned int cs = sum_acc - (kA8 ? 128u : 8u) * 32u;  // every code carried an offset
    if (row_warp) {
      cs = __reduce_add_sync(0xffffffffu, cs);
      if (!one_warp && (tid & 31) == 0 && rloc < rpc) atomicAdd(&s_sum[rloc], cs);
    } else {
      cs += __shfl_xor_sync(0xffffffffu, cs, 1);
      cs += __shfl_xor_sync(0xffffffffu, cs, 2);
      if ((tid & 3) == 0 && rloc < rpc) atomicAdd(&s_sum[rloc], cs);
    }
    if (!one_warp) {
      __syncthreads();
      cs = s_sum[rloc < rpc ? rloc : 0];
    }
    if (active && j == 0) xsum[m] = static_cast<int32_t>(cs);
  }
}

template <typename T, int kLogB, bool kStep, int kOut>
cudaError_t launch_wide_t(const RotQuantArgs& a) {
  const int tpr = a.K / 32;
  int rows = tpr >= 256 ? 1 : 256 / tpr;
  if (rows > kWideRows) rows = kWideRows;
  while (rows > 1 && (a.M + rows - 1) / rows < a.num_sms) rows /= 2;  // few rows: more CTAs, down to one row each
  const int tpb = (rows * tpr + 31) & ~31;  // whole warps: the warp-wide steps take every lane
  rows = tpb / tpr;                         // as the kernel counts them
  auto kern = rotate_quant_wide_kernel<T, kLogB, kStep, kOut>;
  const size_t smem = kLogB > 5 ? static_cast<size_t>(tpb) * 128 : 0;
  if (smem > 40 * 1024) {  // (48 KB without it, the kernel's own few words included)
    constexpr int kMaxSmem = kWideThreads * 128;  // raised once per device to the most any K asks of it
    static std::atomic<unsigned long long> raised{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(raised.load() & bit)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
      if (e != cudaSuccess) return e;
      raised.fetch_or(bit);
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((a.M + rows - 1) / rows));
  cfg.blockDim = dim3(static_cast<unsigned>(tpb));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = a.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // may overlap the previous kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<const T*>(a.x), a.M, a.K, a.inv_sqrt_b, a.step_scale, a.xq,
                                     a.xscale, a.xsum, a.gshift, a.xgsum, a.zero, a.zero_n);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename T, bool kStep, int kOut>
cudaError_t launch_wide_b(const RotQuantArgs& a) {
  switch (a.log_b) {
    case 0: return launch_wide_t<T, 0, kStep, kOut>(a);
    case 1: return launch_wide_t<T, 1, kStep, kOut>(a);
    case 2: return launch_wide_t<T, 2, kStep, kOut>(a);
    case 3: return launch_wide_t<T, 3, kStep, kOut>(a);
    case 4: return launch_wide_t<T, 4, kStep, kOut>(a);
    case 5: return launch_wide_t<T, 5, kStep, kOut>(a);
    case 6: return launch_wide_t<T, 6, kStep, kOut>(a);
    case 7: return launch_wide_t<T, 7, kStep, kOut>(a);
    case 8: return launch_wide_t<T, 8, kStep, kOut>(a);
    case 9: return launch_wide_t<T, 9, kStep, kOut>(a);
    case 10: return launch_wide_t<T, 10, kStep, kOut>(a);
    case 11: return launch_wide_t<T, 11, kStep, kOut>(a);
    default: return launch_wide_t<T, 12, kStep, kOut>(a);
  }
}

template <typename T, int kOut>
cudaError_t launch_wide(const RotQuantArgs& a) {
  return a.mode == 1 ? launch_wide_b<T, true, kOut>(a) : launch_wide_b<T, false, kOut>(a);
}

}  // namespace rq
}  // namespace qvla
