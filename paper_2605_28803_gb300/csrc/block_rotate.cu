// Online data-dependent rotation x' = x . P . BlockDiag(U_1, ..., U_nb) (Sec. 4.1, Eq. 4-5) for a
// layer whose activations cannot take it upstream (layers that share an input but fold different
// U_b, such as Q, K and V).  Float32 products and sums, one rounding to the activation dtype; the
// Hadamard factor and the quantiser then run on x' as for any other layer.
//
// Small batches: one CTA takes 64 rows of one channel block b: it stages U_b (row-major [i][c]) and the 64 gathered input
// rows x[m][perm[b*kB + i]] in shared memory, and each thread accumulates a 4-row x (kB/16)-column patch of
// x'[m][b*kB + c] = sum_i x[m][perm[b*kB + i]] U_b[i][c] in the order i = 0, 1, ..., kB - 1.
//
// The gather takes a 32-byte sector for every value, and the patch a word of shared memory for every two products: at
// 3325 x 10112 (bf16, blocks of 64) that kernel takes 193 us, where memory needs 20 (67 MB each way) and the products 58 at
// 128 a clock and SM.  Large batches therefore take two kernels, 115 us there: a pass that permutes whole rows through
// shared memory (28 us, 4.8 TB/s), and the blocks in place on coalesced tiles (94 us; 41 with blocks of 16).  The second
// is bound by the float32 products: patches of 8 x 4 and staying CTAs with the next tile's loads under way came out equal or
// slower.  816 x 16384 83 and 52 us, f32 3000 x 4096 117 and 53.  Both paths sum in the same order: the same bits.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>
#include <cstdint>

#include "griddep.cuh"
#include "kernels.h"

namespace qvla {
namespace {

constexpr int kRows = 64;  // rows per CTA
constexpr int kBrThreads = 256;

template <typename T>
__device__ __forceinline__ float load_f(const T* p);
template <>
__device__ __forceinline__ float load_f<__half>(const __half* p) {
  return __half2float(*p);
}
template <>
__device__ __forceinline__ float load_f<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}
template <>
__device__ __forceinline__ float load_f<float>(const float* p) {
  return *p;
}

template <typename T>
__device__ __forceinline__ T round_to(float v);
template <>
__device__ __forceinline__ __half round_to<__half>(float v) {
  return __float2half_rn(v);
}
template <>
__device__ __forceinline__ __nv_bfloat16 round_to<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}
template <>
__device__ __forceinline__ float round_to<float>(float v) {
  return v;
}

template <typename T, int kB>
__global__ void __launch_bounds__(kBrThreads) block_rotate_kernel(const T* __restrict__ x, int M, int K,
                                                                   const int32_t* __restrict__ perm,
                                                                   const float* __restrict__ rot, T* __restrict__ out) {
  static_assert(kB % 16 == 0 && kB <= 64, "blocks of 16, 32 or 64 channels");
  constexpr int kC = kB / 16;  // output columns per thread, 16 apart
  __shared__ __align__(16) float su[kB * kB];
  __shared__ float sz[kRows][kB + 1];  // padded: the two row groups of a warp read distinct banks
  const int b = blockIdx.x;
  const int m0 = blockIdx.y * kRows;
  const int t = threadIdx.x;

  // every load is issued before any is used: thread t gathers channel perm[b kB + t % kB] of rows
  // t / kB, t / kB + kRStep, ..., and copies float4 t, t + kBrThreads, ... of U_b
  static_assert(kBrThreads % kB == 0, "a thread's gathered channel is fixed");
  constexpr int kRStep = kBrThreads / kB;
  constexpr int kPer = kRows / kRStep;                     // gathered values per thread
  constexpr int kU4 = kB * kB / 4;                         // float4 of U_b
  constexpr int kUPer = (kU4 + kBrThreads - 1) / kBrThreads;
  const float4* usrc = reinterpret_cast<const float4*>(rot + static_cast<size_t>(b) * kB * kB);
  float4 uv[kUPer];
#pragma unroll
  for (int j = 0; j < kUPer; ++j)
    if (kU4 % kBrThreads == 0 || t + j * kBrThreads < kU4) uv[j] = __ldg(usrc + t + j * kBrThreads);
  const int gi = t % kB, gr = t / kB;
  const int col = __ldg(perm + b * kB + gi);
  float gv[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int m = m0 + gr + j * kRStep;
    gv[j] = m < M ? load_f(x + static_cast<size_t>(m) * K + col) : 0.0f;
  }
#pragma unroll
  for (int j = 0; j < kUPer; ++j)
    if (kU4 % kBrThreads == 0 || t + j * kBrThreads < kU4) reinterpret_cast<float4*>(su)[t + j * kBrThreads] = uv[j];
#pragma unroll
  for (int j = 0; j < kPer; ++j) sz[gr + j * kRStep][gi] = gv[j];
  __syncthreads();

  const int rg = t >> 4, cg = t & 15;  // rows 4 rg .. 4 rg + 3, columns cg + 16 j
  float acc[4][kC];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int j = 0; j < kC; ++j) acc[a][j] = 0.0f;
#pragma unroll 4
  for (int i = 0; i < kB; ++i) {
    float z[4], u[kC];
#pragma unroll
    for (int a = 0; a < 4; ++a) z[a] = sz[4 * rg + a][i];
#pragma unroll
    for (int j = 0; j < kC; ++j) u[j] = su[i * kB + cg + 16 * j];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int j = 0; j < kC; ++j) acc[a][j] = fmaf(z[a], u[j], acc[a][j]);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int m = m0 + 4 * rg + a;
    if (m >= M) continue;
    T* dst = out + static_cast<size_t>(m) * K + b * kB + cg;
#pragma unroll
    for (int j = 0; j < kC; ++j) dst[16 * j] = round_to<T>(acc[a][j]);
  }
}

// ---- many rows: the permutation as a pass of its own, then the blocks in place -----------------------------------------

constexpr int kPermThreads = 256;
constexpr int kAhead = 3;         // 16-byte pieces of a row that a thread has in flight
constexpr int kTileRows = 128;    // rows of a CTA of the second kernel
constexpr int kTileChans = 64;    // its channels: 64 / kB blocks
constexpr int kTileThreads = 128;

// out[m][c] = x[m][perm[c]].  A CTA stages its rows and gathers from shared memory; 16-bit types keep two rows in the
// halves of a word, so that one load gathers for both.
template <typename T>
__global__ void __launch_bounds__(kPermThreads) permute_rows_kernel(const T* __restrict__ x, int M, int K,
                                                                     const int32_t* __restrict__ perm, T* __restrict__ out) {
  extern __shared__ __align__(16) uint32_t words[];  // [K]
  constexpr int kPair = sizeof(T) == 2 ? 2 : 1;
  griddep_launch_dependents();
  const int m = blockIdx.x * kPair;
  const T* src = x + static_cast<size_t>(m) * K;
  T* dst = out + static_cast<size_t>(m) * K;
  constexpr int kChans = kPair == 2 ? 8 : 4;  // channels of 16 bytes
  constexpr int kStep = kPermThreads * kChans;
  const bool two = kPair == 2 && m + 1 < M;
  int4 p[kAhead][kChans / 4];
#pragma unroll
  for (int j = 0; j < kAhead; ++j) {  // the first indices are on their way while the rows are staged
    const int c = (threadIdx.x + j * kPermThreads) * kChans;
#pragma unroll
    for (int k = 0; k < kChans / 4; ++k)
      if (c < K) p[j][k] = __ldg(reinterpret_cast<const int4*>(perm + c) + k);
  }
  for (int c0 = threadIdx.x * kChans; c0 < K; c0 += kAhead * kStep) {
    uint4 a[kAhead], b[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int c = c0 + j * kStep;
      a[j] = c < K ? __ldg(reinterpret_cast<const uint4*>(src + c)) : make_uint4(0, 0, 0, 0);
      b[j] = two && c < K ? __ldg(reinterpret_cast<const uint4*>(src + K + c)) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int c = c0 + j * kStep;
      if (c >= K) break;
      uint4* w = reinterpret_cast<uint4*>(words + c);
      if constexpr (kPair == 2) {
        w[0] = make_uint4(__byte_perm(a[j].x, b[j].x, 0x5410), __byte_perm(a[j].x, b[j].x, 0x7632),
                          __byte_perm(a[j].y, b[j].y, 0x5410), __byte_perm(a[j].y, b[j].y, 0x7632));
        w[1] = make_uint4(__byte_perm(a[j].z, b[j].z, 0x5410), __byte_perm(a[j].z, b[j].z, 0x7632),
                          __byte_perm(a[j].w, b[j].w, 0x5410), __byte_perm(a[j].w, b[j].w, 0x7632));
      } else {
        w[0] = a[j];
      }
    }
  }
  __syncthreads();
  for (int c0 = threadIdx.x * kChans; c0 < K; c0 += kAhead * kStep) {
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int c = c0 + j * kStep;
      if (c >= K) break;
      const int4 q = p[j][0];
      uint32_t w[kChans];
      w[0] = words[q.x], w[1] = words[q.y], w[2] = words[q.z], w[3] = words[q.w];
      if constexpr (kPair == 2) {
        const int4 r = p[j][1];
        w[4] = words[r.x], w[5] = words[r.y], w[6] = words[r.z], w[7] = words[r.w];
        *reinterpret_cast<uint4*>(dst + c) = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410),
                                                        __byte_perm(w[4], w[5], 0x5410), __byte_perm(w[6], w[7], 0x5410));
        if (two)
          *reinterpret_cast<uint4*>(dst + K + c) = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632),
                                                              __byte_perm(w[4], w[5], 0x7632), __byte_perm(w[6], w[7], 0x7632));
      } else {
        *reinterpret_cast<uint4*>(dst + c) = make_uint4(w[0], w[1], w[2], w[3]);
      }
#pragma unroll
      for (int k = 0; k < kChans / 4; ++k)
        if (c + kAhead * kStep < K) p[j][k] = __ldg(reinterpret_cast<const int4*>(perm + c + kAhead * kStep) + k);
    }
  }
}

// Two values of rows 2 p and 2 p + 1 as floats.
template <typename T>
__device__ __forceinline__ float2 pair_f(uint32_t w);
template <>
__device__ __forceinline__ float2 pair_f<__half>(uint32_t w) {
  return __half22float2(*reinterpret_cast<__half2*>(&w));
}
template <>
__device__ __forceinline__ float2 pair_f<__nv_bfloat16>(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}

// y[m][b kB + c] = sum_i y[m][b kB + i] U_b[i][c] in place: a CTA reads its 128 x 64 tile whole before it writes it.  A thread
// sums 8 rows x 8 columns, two rows to an instruction, each in the order i = 0 .. kB - 1 as above.  The tile is kept
// transposed, 16-bit types as they are with two rows to a word: then shared memory gives 64 bytes for 64 products.
template <typename T, int kB>
__global__ void __launch_bounds__(kTileThreads, 4) rotate_tile_kernel(T* y, int M, int K, const float* __restrict__ rot) {
  constexpr bool k16 = sizeof(T) == 2;
  constexpr int kW = k16 ? kTileRows / 2 : kTileRows;       // words of a channel
  __shared__ __align__(16) uint32_t sz[kTileChans * kW];    // [i][word]; the words of channel i moved by 4 (i / 8), see below
  __shared__ __align__(16) float su[kTileChans * kB];       // [block][i][c]
  constexpr int kPer16 = 16 / static_cast<int>(sizeof(T));  // channels of a 16-byte piece
  constexpr int kPieces = kTileChans / kPer16;              // pieces of a row's tile
  constexpr int kRowsEach = k16 ? 2 : 1;                    // rows a thread stages together
  constexpr int kLoads = kTileRows * kPieces / kTileThreads / kRowsEach;
  const int t = threadIdx.x;
  const int ch0 = blockIdx.x * kTileChans, m0 = blockIdx.y * kTileRows;

  const float4* usrc = reinterpret_cast<const float4*>(rot + static_cast<size_t>(ch0) * kB);  // U_b at b kB kB = ch0 kB
#pragma unroll
  for (int j = 0; j < kTileChans * kB / 4 / kTileThreads; ++j)
    reinterpret_cast<float4*>(su)[t + j * kTileThreads] = __ldg(usrc + t + j * kTileThreads);
  griddep_wait();  // y is the permutation's output
  griddep_launch_dependents();
  const int ck = t % kPieces, r0 = t / kPieces;
  uint4 in[kLoads][kRowsEach];
#pragma unroll
  for (int j = 0; j < kLoads; ++j)
#pragma unroll
    for (int e = 0; e < kRowsEach; ++e) {
      const int m = m0 + (r0 + j * (kTileThreads / kPieces)) * kRowsEach + e;
      in[j][e] = m < M ? *reinterpret_cast<const uint4*>(y + static_cast<size_t>(m) * K + ch0 + ck * kPer16) : make_uint4(0, 0, 0, 0);
    }
  // the pieces that a warp stores at once are 8 channels (or 4) apart: moved by 4 words for each 8 they fall on other banks
#pragma unroll
  for (int j = 0; j < kLoads; ++j) {
    const int w = r0 + j * (kTileThreads / kPieces);
    const uint32_t* a = reinterpret_cast<const uint32_t*>(&in[j][0]);
    const int i0 = ck * kPer16;
    uint32_t* d = sz + i0 * kW + (w ^ (((i0 >> 3) & 7) << 2));
    if constexpr (k16) {
      const uint32_t* b = reinterpret_cast<const uint32_t*>(&in[j][1]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        d[(2 * k) * kW] = __byte_perm(a[k], b[k], 0x5410);
        d[(2 * k + 1) * kW] = __byte_perm(a[k], b[k], 0x7632);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) d[k * kW] = a[k];
    }
  }
  __syncthreads();

  // rows 8 rg .. 8 rg + 7; columns c0 .. c0 + 3 and c1 .. c1 + 3, the halves of 8 cg .. 8 cg + 7, the upper one first for
  // cg >= 4 (8 threads read 128 distinct bytes of a row of U at a time)
  const int rg = t >> 3, cg = t & 7, up = cg >> 2;
  const int blk = 8 * cg / kB;
  const int c0 = (8 * cg) % kB + 4 * up, c1 = (8 * cg) % kB + 4 - 4 * up;
  float2 acc[4][8];  // [rows 2 a, 2 a + 1][column]
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[a][j] = make_float2(0.0f, 0.0f);
  const float* ub = su + blk * kB * kB;
#pragma unroll 1
  for (int i8 = 0; i8 < kB; i8 += 8) {
    const int at = blk * kB + i8, move = ((at >> 3) & 7) << 2;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 u0 = *reinterpret_cast<const float4*>(ub + (i8 + k) * kB + c0);
      const float4 u1 = *reinterpret_cast<const float4*>(ub + (i8 + k) * kB + c1);
      const uint32_t* zr = sz + (at + k) * kW;
      float2 z[4];
      if constexpr (k16) {
        const uint4 w = *reinterpret_cast<const uint4*>(zr + ((4 * rg) ^ move));
        z[0] = pair_f<T>(w.x), z[1] = pair_f<T>(w.y), z[2] = pair_f<T>(w.z), z[3] = pair_f<T>(w.w);
      } else {
        const float4 a = *reinterpret_cast<const float4*>(zr + ((8 * rg) ^ move));
        const float4 b = *reinterpret_cast<const float4*>(zr + ((8 * rg + 4) ^ move));
        z[0] = make_float2(a.x, a.y), z[1] = make_float2(a.z, a.w), z[2] = make_float2(b.x, b.y), z[3] = make_float2(b.z, b.w);
      }
      const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a][j] = __ffma2_rn(z[a], make_float2(u[j], u[j]), acc[a][j]);
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int m = m0 + 8 * rg + r;
    if (m >= M) continue;
    struct __align__(4 * sizeof(T)) Four {
      T v[4];
    } lo, hi;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T a = round_to<T>(r % 2 ? acc[r / 2][j].y : acc[r / 2][j].x);
      const T b = round_to<T>(r % 2 ? acc[r / 2][4 + j].y : acc[r / 2][4 + j].x);
      lo.v[j] = up ? b : a;
      hi.v[j] = up ? a : b;
    }
    Four* dst = reinterpret_cast<Four*>(y + static_cast<size_t>(m) * K + ch0 + 8 * cg);
    dst[0] = lo;
    dst[1] = hi;
  }
}

template <typename T>
cudaError_t launch_two(const T* x, int M, int K, const int32_t* perm, const float* rot, int block, T* out, cudaStream_t stream) {
  auto kern = permute_rows_kernel<T>;
  const size_t smem = static_cast<size_t>(K) * 4;
  if (smem > 48 * 1024) {  // raised once per device to the largest K's
    static std::atomic<unsigned long long> raised{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(raised.load() & bit)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * 4);
      if (e != cudaSuccess) return e;
      raised.fetch_or(bit);
    }
  }
  constexpr int kPair = sizeof(T) == 2 ? 2 : 1;
  kern<<<(M + kPair - 1) / kPair, kPermThreads, smem, stream>>>(x, M, K, perm, out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(K / kTileChans, (M + kTileRows - 1) / kTileRows);
  cfg.blockDim = dim3(kTileThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // U_b is loaded while the permutation ends
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  switch (block) {
    case 16: e = cudaLaunchKernelEx(&cfg, rotate_tile_kernel<T, 16>, out, M, K, rot); break;
    case 32: e = cudaLaunchKernelEx(&cfg, rotate_tile_kernel<T, 32>, out, M, K, rot); break;
    case 64: e = cudaLaunchKernelEx(&cfg, rotate_tile_kernel<T, 64>, out, M, K, rot); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// Two kernels from 2^21 values and rows of 1024 channels on: there they are faster for every block and type (us, one kernel and
// two, blocks of 64: bf16 1171 x 2048 16.4 and 16.1, 2441 x 2048 32.8 and 22.3, 3320 x 1024 21.3 and 16.4, 146 x 16384 23.6
// and 20.7; f32 1171 x 2048 27.9 and 17.7; blocks of 16: bf16 2343 x 1024 11.1 and 7.7, f32 1171 x 2048 13.1 and 12.5).
// Below, the second launch costs more than it saves (830 x 2048 12.7 and 15.7), and short rows stay in L1, where the gather
// is cheap (6640 x 512 f32 14.9 and 17.1, blocks of 16).
bool takes_two(const void* x, int M, int K, const void* out) {
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(out)) & 15u) return false;  // 16-byte loads and stores
  return K >= 1024 && static_cast<long long>(M) * K >= (1 << 21);
}

template <typename T>
cudaError_t launch_t(const void* x, int M, int K, const int32_t* perm, const float* rot, int block, void* out,
                     cudaStream_t stream) {
  const T* xt = static_cast<const T*>(x);
  T* ot = static_cast<T*>(out);
  if (takes_two(x, M, K, out)) return launch_two<T>(xt, M, K, perm, rot, block, ot, stream);
  const dim3 grid(K / block, (M + kRows - 1) / kRows);
  switch (block) {
    case 16: block_rotate_kernel<T, 16><<<grid, kBrThreads, 0, stream>>>(xt, M, K, perm, rot, ot); break;
    case 32: block_rotate_kernel<T, 32><<<grid, kBrThreads, 0, stream>>>(xt, M, K, perm, rot, ot); break;
    case 64: block_rotate_kernel<T, 64><<<grid, kBrThreads, 0, stream>>>(xt, M, K, perm, rot, ot); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_block_rotate(const void* x, int xdt, int M, int K, const int32_t* perm, const float* rot, int block,
                                void* out, cudaStream_t stream) {
  if (M == 0) return cudaSuccess;
  if (block <= 0 || K % block != 0) return cudaErrorInvalidValue;
  switch (xdt) {
    case 0: return launch_t<__half>(x, M, K, perm, rot, block, out, stream);
    case 1: return launch_t<__nv_bfloat16>(x, M, K, perm, rot, block, out, stream);
    case 2: return launch_t<float>(x, M, K, perm, rot, block, out, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qvla
