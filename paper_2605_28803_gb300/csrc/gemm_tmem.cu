// W4A4 / W4A8 GEMM for batches of more than 128 tokens and for gated layers (Sec. 4.2, Eq. 7): CTA pairs, the expanded
// weights in TMEM.
//
// The product is taken weight-major: D[weight row, token] = W X^T, one 2-SM tcgen05.mma (cta_group::2, M = 256 weight
// rows, N = bn tokens) per 32 codes.  The packed weights are expanded to offset-E4M3 bytes (code q as the byte q + 8)
// straight into TMEM as the MMA's A operand, so the expanded tile is never written to or read from shared memory;
// operand B is the rotate-quantise kernel's operand bytes, TMA-loaded with the 128-byte swizzle.  Per k-block of 128
// codes and SM, shared memory then carries 8 KB of packed weights and 64 bn bytes of activations in and out (40 KB at
// bn = 192) against 384 cycles of tensor work.  Accumulation is exact (see gemm_kernel.cuh), so the outputs are the
// bits of the other GEMM kernels of the library.
//
// One persistent CTA pair per SM pair.  Warp roles of a CTA:
//   warps 0-7    epilogue, two warps per TMEM lane quadrant on alternate 32-token chunks: TMEM -> registers ->
//                dequantise -> transposed into shared memory -> TMA store (stores straight from registers, 64 bytes of
//                a token row per warp, took 52 of the 205 us of 8192 x 2048 -> 16384)
//   warps 8-23   converters, four groups of four (one warp per TMEM lane quadrant), two groups for the even ring stages
//                and two for the odd ones, half a stage each: packed weights -> registers -> E4M3 bytes in TMEM
//   warp  24     TMEM allocation; in the pair's leader one thread issues the MMAs and the commits
//   warp  25     one thread issues the TMA loads of the activation tiles
//   warp  26     one thread issues the TMA loads of the packed weights
// (warp 27 fills the last warpgroup: the register split below is per warpgroup.)  The issuing warps run their loops
// whole and elect one thread around the issues: a loop run by one lane alone costs a loop over the active lanes at every
// TMA or tensor-core instruction (measured: 1080 against 760 cycles a k-block).
// Every ring stage holds two activation tiles (two k-blocks, or the two planes of one k-block of 8-bit codes) and the
// weights that multiply them: 8 MMAs.  A round of wait, TMA loads and expected-bytes arrival takes about 450 cycles
// whatever the loads' size, so a round per k-block would bound the kernel at that (816 x 16384 -> 2048 at bn = 128: 1035
// cycles a k-block with every role on one k-block per round, 430 now).
// TMEM (512 columns): two accumulators of bn columns, then a ring of weight stages (32 columns per k-block); a stage's
// k-blocks are filled and released one by one, which hides the release-refill latency (about 1400 cycles) at bn = 192,
// where the ring holds four k-blocks.
//
// GEMM alone, in us, token-major kernel before and this one: 816 x 2048 -> 2 x 16384 gated 60.4 and 42.3 (2590 TFLOP/s
// of the integer product); 816 x 16384 -> 2048 38.0 and 26.2; 8192 x 2048 -> 16384 240 and 146 (3770 TFLOP/s); 3200 x
// 16384 -> 2048 104.6 and 57.4 (3740 TFLOP/s); 8-bit codes, 816 x 2048 -> 2 x 16384 gated 79 and 63.  Packed 4-bit codes,
// expanded by the converters next to the weights: 777 x 4096 -> 1024 18.0 and 12.5, 5781 x 3712 -> 7392 142 and 121, 816 x
// 2048 -> 2 x 16384 gated 72 and 59, 50 x 2048 -> 2 x 4096 gated 15.1 and 7.9; a k-block costs the converters 235 to 290 ns
// there (the codes fetched before the wait for the TMEM stage, and the proxy fence moved up to the stores, were slower: 40
// against 34 us at 200 x 16384 -> 2048).  Bound now by the
// issue round of the MMA warp (about 430 cycles a k-block up to bn = 160) and the refill of the TMEM stages (about 470 at
// 192), against 384 cycles of tensor work at bn = 192.
#include "gemm_kernel.cuh"

namespace qvla {
namespace {

constexpr int kTmEpiWarps = 8, kTmConv = 8, kTmMma = 24, kTmTmaX = 25, kTmTmaW = 26;  // first warp of each role
constexpr int kTmGroups = 4;  // converter groups
constexpr int kTmEpiThreads = kTmEpiWarps * 32;
constexpr int kTmThreads = 28 * 32;
// Registers: 72 a thread at launch (896 x 72 = 64512); the roles then take 256 x 120 + 512 x 56 + 128 x 40 = 64512.  The
// instances for operand bytes of 4-bit codes spill 6 bytes a thread (-Xptxas -v), the others none.
constexpr int kTmRegsEpi = 120, kTmRegsConv = 56, kTmRegsOther = 40;
static_assert(256 * kTmRegsEpi + 512 * kTmRegsConv + 128 * kTmRegsOther <= kTmThreads * 72, "register split");
constexpr int kTmMaxBn = 192;          // 2 x 192 accumulator columns leave two weight stages of two k-blocks
constexpr int kTmMaxStages = 8;
constexpr int kTmRaw = kBM * kBK / 2;  // bytes of packed weights per CTA and k-block
constexpr int kTmOut = kBM * 32 * 2;    // bytes of an output chunk: 32 tokens x 128 channels
constexpr int kTmOutBytes = 4 * kTmOut;  // two chunks for each half of the epilogue warps
constexpr int kTmSmem = 180 * 1024;    // rings

struct TmParams {
  const float* xscale;  // [M]
  const int32_t* xsum;  // [M]
  const float* wscale;  // [N]
  const float* wcorr;   // [N] 8 x (int8 activations: 128 x) the weights' code sums
  const float* bias;    // [N]
  int32_t* acc;
  int M, N, nkb;
  int bn;                  // tokens per tile: a multiple of 32, at most kTmMaxBn
  int stages, stages_a;    // depths of the rings (weights and activations alike) and of the weight stages in TMEM
  int tiles_m, tiles_n;    // token tiles; 256-row weight tiles
  // a tile's k-blocks in `parts` work units (1 = whole tiles); partials [tile][part][CTA][bn / 4][128] float4,
  // part_cnt [tile][CTA] the finished units (zero at launch, left zero)
  int parts;
  float* part_ws;
  int* part_cnt;
  float kconst;
};

// 2-SM MMA with A in TMEM; the descriptor of B as its two halves.
__device__ __forceinline__ void mma_e4m3_pair_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi,
                                                 uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 b;\nsetp.ne.b32 p, %5, 0;\nmov.b64 b, {%2, %3};\n"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], [%1], b, %4, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The four epilogue warps of one half (0 or 1) meet.
__device__ __forceinline__ void tm_half_sync(int half) {
  asm volatile("bar.sync %0, %1;" ::"r"(kEpiBarrier + 1 + half), "n"(kTmEpiThreads / 2) : "memory");
}
__device__ __forceinline__ void tm_epi_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(kEpiBarrier), "n"(kTmEpiThreads) : "memory");
}

// kGated: the weight tile is 128 hidden units; CTA r of the pair takes units 64 r .. 64 r + 63, gate and up rows, in
// TMEM lanes 32 q + i (gate of unit 64 r + 16 q + i) and 32 q + 16 + i (its up row), i < 16.
// kPlanes: operand tiles of the activations per k-block (2: the high and low nibbles of 8-bit codes).
// kPacked: the activations are packed int4 codes; the converters of a k-block expand its tokens too, into tiles as many and as
// long in use as the weight stages in TMEM.
template <bool kGated, int kPlanes, bool kPacked, typename OutT>
__global__ void __launch_bounds__(kTmThreads, 1) gemm_tmem_kernel(const __grid_constant__ CUtensorMap tmap_x,
                                                                  const __grid_constant__ CUtensorMap tmap_w,
                                                                  const __grid_constant__ CUtensorMap tmap_y, TmParams p) {
  constexpr int kKb = 2 / kPlanes;  // k-blocks per ring stage
  static_assert(!kPacked || kPlanes == 1, "packed 4-bit codes");
  extern __shared__ uint8_t dyn_smem[];
  uint8_t* const smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bar_rfull[kTmMaxStages];   // packed weights landed
  __shared__ __align__(8) uint64_t bar_rempty[kTmMaxStages];  // every converter warp is done with them
  // leader: both CTAs' weights of the stage's k-block h are in TMEM; for h = 0 also both CTAs' activation tiles landed
  __shared__ __align__(8) uint64_t bar_full[kTmMaxStages][kKb];
  // the MMAs have read the weights of k-block h of stage s from TMEM; for the last h also the stage's activation tiles
  __shared__ __align__(8) uint64_t bar_empty[kTmMaxStages][kKb];
  __shared__ __align__(8) uint64_t bar_tfull[2], bar_tempty[2];
  __shared__ __align__(8) uint64_t bar_done;
  __shared__ uint32_t s_tmem_base;
  __shared__ int s_epi_abort, s_last;
  __shared__ __align__(16) float s_xs[kTmMaxBn], s_cm[kTmMaxBn];  // this tile's tokens: scale, - zero-point correction

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int bn = p.bn, nkb = p.nkb, S = p.stages, SA = p.stages_a, parts = p.parts;
  const int units = p.tiles_m * p.tiles_n * parts;
  const int unit0 = static_cast<int>(blockIdx.x >> 1), ustep = static_cast<int>(gridDim.x >> 1);
  const int btile = bn / 2 * kBK;               // bytes of one activation tile of this CTA
  uint8_t* const out_smem = smem;               // [half][2][kTmOut] output chunks
  uint8_t* const ring_b = smem + kTmOutBytes;   // [S (packed codes: SA)][2][bn / 2][128], 128-byte swizzled
  uint8_t* const ring_r = ring_b + (kPacked ? SA : S) * 2 * btile;  // [S][kKb][128][64] (gated: [S][gate, up][kKb][64][64]), 64-byte swizzled
  uint8_t* const ring_x = ring_r + S * kKb * kTmRaw;  // packed codes: [S][2][bn / 2][64]

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&bar_rfull[s]), kPacked ? 2 : 1);  // the expected bytes, of packed activations too
      mbar_init(smem_u32(&bar_rempty[s]), 2 * kTmGroups);
      for (int h = 0; h < kKb; ++h) {  // the expected bytes, the k-block's converter warps of both CTAs
        mbar_init(smem_u32(&bar_full[s][h]), (h == 0 && !kPacked ? 1 : 0) + 4 * kTmGroups / kKb);
        mbar_init(smem_u32(&bar_empty[s][h]), 1);
      }
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&bar_tfull[i]), 1);
      mbar_init(smem_u32(&bar_tempty[i]), 2 * kTmEpiWarps);  // the epilogue warps of both CTAs
    }
    mbar_init(smem_u32(&bar_done), 1);
    mbar_init_fence();
    s_epi_abort = 0;
  }
  if (warp == kTmMma) tmem_alloc_pair<512>(smem_u32(&s_tmem_base));
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before any arrival crosses the pair
  tc_fence_after();
  const uint32_t tmem = s_tmem_base;
  const uint32_t tmem_a = tmem + static_cast<uint32_t>(2 * bn);  // the weight stages
  if (threadIdx.x == 0) griddep_launch_dependents();

  // work unit u: weight tile tb, token tile ta, k-blocks [ka, kz)
  auto unit_at = [&](int u, int& tile, int& ta, int& tb, int& ka, int& kz) {
    tile = u / parts;
    const int part = u - tile * parts;
    ta = tile % p.tiles_m;
    tb = tile / p.tiles_m;
    ka = nkb * part / parts;
    kz = nkb * (part + 1) / parts;
  };

  if (warp >= kTmMma) {
    setmaxnreg_dec<kTmRegsOther>();
    if (warp == kTmTmaX) {
      // ------------------------------------------------------------------ activation tiles
      // (the whole warp runs the loop, so that its values are uniform; one thread issues)
      {
        tma_prefetch_desc(&tmap_x);
        bool ok = *const_cast<volatile int*>(&g_debug_hold_loads) == 0;  // test hook: issue nothing
        griddep_wait();
        int it = 0, s = 0;
        uint32_t ph = 0;
        for (int u = unit0; u < units && ok; u += ustep) {
          int tile, ta, tb, ka, kz;
          unit_at(u, tile, ta, tb, ka, kz);
          const int row = ta * bn + static_cast<int>(rank) * (bn / 2);
          for (int kb = ka; kb < kz; kb += kKb, ++it) {
            if constexpr (kPacked) {  // this CTA's codes, for its own converters
              if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_rempty[s]), ph ^ 1u))) { ok = false; break; }
              const uint32_t bar = smem_u32(&bar_rfull[s]), dst = smem_u32(ring_x + s * btile);
              const bool two = kb + 1 < kz;
              if (elect_one()) {
                mbar_arrive_expect_tx(bar, static_cast<uint32_t>((two ? 2 : 1) * (btile / 2)));
                tma_load_2d(dst, &tmap_x, kb * (kBK / 2), row, bar);
                if (two) tma_load_2d(dst + btile / 2, &tmap_x, (kb + 1) * (kBK / 2), row, bar);
              }
              __syncwarp();
              if (++s == S) { s = 0; ph ^= 1u; }
              continue;
            }
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_empty[s][kKb - 1]), ph ^ 1u))) { ok = false; break; }
            // both CTAs' tiles complete on the leader's barrier; a unit's last stage may hold one k-block only
            const uint32_t fb = smem_u32(&bar_full[s][0]);
            const bool two = kPlanes == 2 || kb + 1 < kz;
            const uint32_t lead = mapa_shared(fb, 0);
            const uint32_t dst = smem_u32(ring_b + s * 2 * btile);
            if (elect_one()) {
              if (rank == 0) mbar_arrive_expect_tx(fb, static_cast<uint32_t>((two ? 4 : 2) * btile));
              tma_load_2d_pair(dst, &tmap_x, kb * kPlanes * kBK, row, lead);
              if (two) tma_load_2d_pair(dst + btile, &tmap_x, (kb * kPlanes + 1) * kBK, row, lead);
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1u; }
          }
        }
        // before leaving, let every load land: the MMAs that read a stage release it
        for (int i = 0; i < S && i < it; ++i) {
          if (--s < 0) { s = S - 1; ph ^= 1u; }
          if constexpr (kPacked) {
            ok = ok && mbar_wait(smem_u32(&bar_rfull[s]), ph);
          } else {
            ok = ok && mbar_wait(smem_u32(&bar_empty[s][kKb - 1]), ph);  // (after a time-out no MMA will release the rest)
          }
        }
      }
      __syncwarp();
    } else if (warp == kTmTmaW) {
      // ------------------------------------------------------------------ packed weights (no earlier kernel writes them)
      {
        tma_prefetch_desc(&tmap_w);
        bool ok = *const_cast<volatile int*>(&g_debug_hold_loads) == 0;
        int it = 0, s = 0;
        uint32_t ph = 0;
        for (int u = unit0; u < units && ok; u += ustep) {
          int tile, ta, tb, ka, kz;
          unit_at(u, tile, ta, tb, ka, kz);
          for (int kb = ka; kb < kz; kb += kKb, ++it) {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_rempty[s]), ph ^ 1u))) { ok = false; break; }
            const uint32_t bar = smem_u32(&bar_rfull[s]);
            const uint32_t dst = smem_u32(ring_r + s * kKb * kTmRaw);
            if (elect_one()) {  // (past a unit's last k-block the box reads the next chunk, which nothing uses)
              mbar_arrive_expect_tx(bar, kKb * kTmRaw);
              if constexpr (kGated) {  // 64 gate rows, then their 64 up rows
                tma_load_3d(dst, &tmap_w, 0, 64 * static_cast<int>(rank), 2 * tb * nkb + kb, bar);
                tma_load_3d(dst + kKb * kTmRaw / 2, &tmap_w, 0, 64 * static_cast<int>(rank), (2 * tb + 1) * nkb + kb, bar);
              } else {
                tma_load_3d(dst, &tmap_w, 0, 0, (2 * tb + static_cast<int>(rank)) * nkb + kb, bar);
              }
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1u; }
          }
        }
        for (int i = 0; i < S && i < it; ++i) {  // before leaving, let every load land
          if (--s < 0) { s = S - 1; ph ^= 1u; }
          mbar_wait(smem_u32(&bar_rfull[s]), ph);
        }
      }
      __syncwarp();
    } else if (warp == kTmMma) {
      // ------------------------------------------------------------------ MMA issuer
      if (rank == 0) {
        const uint32_t idesc = idesc_e4m3_f32(2 * kBM, bn);
        const uint32_t desc_hi = static_cast<uint32_t>(smem_desc_sw128(0) >> 32), desc_lo = static_cast<uint32_t>(smem_desc_sw128(0));
        const uint32_t b0 = smem_u32(ring_b), b_stage = static_cast<uint32_t>(2 * btile) >> 4, b_tile = static_cast<uint32_t>(btile) >> 4;
        int s = 0, sa = 0, tile_iter = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int u = unit0; u < units && ok; u += ustep, ++tile_iter) {
          int tile, ta, tb, ka, kz;
          unit_at(u, tile, ta, tb, ka, kz);
          const int buf = tile_iter & 1;
          if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_tempty[buf]), (static_cast<uint32_t>(tile_iter >> 1) & 1u) ^ 1u))) break;
          tc_fence_after();
          const uint32_t d = tmem + static_cast<uint32_t>(buf * bn);
          for (int kb = ka; kb < kz; kb += kKb) {
            const uint32_t a = tmem_a + static_cast<uint32_t>(sa * kKb * 32);
            const uint32_t b = (desc_lo | (b0 >> 4)) + static_cast<uint32_t>(kPacked ? sa : s) * b_stage;
#pragma unroll
            for (int h = 0; h < kKb; ++h) {
              // A unit's last stage may hold one k-block.  The converters fill and announce its second one all the same
              // (bytes that no MMA reads): it is waited for before it is released, or a late store of theirs could land
              // on the slot's next weights, which with an odd SA other warps write.
              const bool real = h == 0 || kb + h < kz;
              if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_full[s][h]), ph))) { ok = false; break; }
              tc_fence_after();
              const uint32_t empty = smem_u32(&bar_empty[s][h]);
              if (elect_one()) {
                if (real) {
#pragma unroll
                  for (int i = 0; i < 4 * kPlanes; ++i) {  // (a k-block's planes meet the same weights)
                    const int t = h + i / 4, kk = i % 4;
                    mma_e4m3_pair_ts(d, a + static_cast<uint32_t>(32 * h + kk * 8),
                                     b + static_cast<uint32_t>(t) * b_tile + static_cast<uint32_t>(kk * 2), desc_hi, idesc,
                                     (kb != ka || h != 0 || i != 0) ? 1u : 0u);
                  }
                }
                mma_commit_pair(empty, 3);
              }
            }
            if (!ok) break;
            if (++s == S) { s = 0; ph ^= 1u; }
            if (++sa == SA) sa = 0;
          }
          if (!ok) break;
          if (elect_one()) mma_commit_pair(smem_u32(&bar_tfull[buf]), 3);
          __syncwarp();
        }
        if (elect_one()) {
          mma_commit_pair(smem_u32(&bar_done), 1);  // every MMA issued above has completed once this flips
          mbar_wait(smem_u32(&bar_done), 0);
        }
      }
      __syncwarp();
    }
  } else if (warp >= kTmConv) {
    // ------------------------------------------------------------------ converters
    setmaxnreg_dec<kTmRegsConv>();
    const int quad = warp & 3;  // the TMEM lanes this warp may write: 32 quad .. 32 quad + 31
    const int group = (warp - kTmConv) >> 2;
    // this group's part of a stage: kPieces 16-byte pieces (32 codes) of every row, from piece `first` of k-block `half`;
    // this lane's row lies under the 64-byte swizzle
    constexpr int kPieces = 2 * kKb;
    const int half = kKb == 2 ? group & 1 : 0, first = kKb == 2 ? 0 : 2 * (group & 1);
    const int row = kGated ? quad * 16 + (lane & 15) : quad * 32 + lane;
    const int x16 = (row >> 1) & 3;
    const uint8_t* const src0 = ring_r + row * 64 + (kGated ? (lane >> 4) * (kKb * kTmRaw / 2) + half * (kTmRaw / 2) : half * kTmRaw);
    const uint32_t dst0 = tmem_a + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(half * 32 + first * 8);
    // Ring position: stage s with its phase ph; the TMEM stage sa, free once the MMAs have read ring stage se (SA stages
    // earlier) in phase pe.  A warp takes every second stage.  Its parity waits cannot be a phase behind: when it waits
    // for its stage j, its wait at j - 2 has shown stage j - 2 - SA multiplied, and with S >= SA + 2 the earlier uses of
    // both barriers (stages j - S and j - SA - S) lie no later than that.
    int s = 0, sa = 0, se = S - SA;
    uint32_t ph = 0, pe = 1;
    auto advance = [&]() {
      if (++s == S) { s = 0; ph ^= 1u; }
      if (++sa == SA) sa = 0;
      if (++se == S) { se = 0; pe ^= 1u; }
    };
    uint4 v[kPieces];
    auto load = [&]() {  // this warp's part of ring stage s, once it has landed
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_rfull[s]), ph))) return false;
#pragma unroll
      for (int c = 0; c < kPieces; ++c)
        v[c] = *reinterpret_cast<const uint4*>(src0 + s * (kKb * kTmRaw) + (((first + c) ^ x16) << 4));
      return true;
    };
    int stages_left = 0;
    for (int u = unit0; u < units; u += ustep) {
      int tile, ta, tb, ka, kz;
      unit_at(u, tile, ta, tb, ka, kz);
      stages_left += (kz - ka + kKb - 1) / kKb;
    }
    if (group >> 1) {
      advance();
      --stages_left;
    }
    bool ok = stages_left > 0 && load();
    for (; ok && stages_left > 0; stages_left -= 2) {
      uint32_t o[8 * kPieces];
#pragma unroll
      for (int c = 0; c < kPieces; ++c) {
        int4x8_to_e4m3_offset(v[c].x, o[8 * c], o[8 * c + 1]);
        int4x8_to_e4m3_offset(v[c].y, o[8 * c + 2], o[8 * c + 3]);
        int4x8_to_e4m3_offset(v[c].z, o[8 * c + 4], o[8 * c + 5]);
        int4x8_to_e4m3_offset(v[c].w, o[8 * c + 6], o[8 * c + 7]);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_empty[se][half]), pe))) break;
      tc_fence_after();
      __syncwarp();
      const uint32_t dst = dst0 + static_cast<uint32_t>(sa * kKb * 32);
      if constexpr (kPieces == 4) {
        tmem_st32(dst, o);
      } else {
        tmem_st16(dst, o);
      }
      if constexpr (kPacked) {  // this k-block's tokens: a thread per 16 bytes (32 codes) of a row
        const uint8_t* const xs = ring_x + s * btile + half * (btile / 2);
        uint8_t* const xd = ring_b + sa * 2 * btile + half * btile;
#pragma unroll 1
        for (int i = (warp & 3) * 32 + lane; i < bn * 2; i += 128) {
          const uint4 c = *reinterpret_cast<const uint4*>(xs + i * 16);
          const int r = i >> 2, q = (2 * i) & 6;
          store_chunk(xd + r * 128, (q ^ (r & 7)) << 4, ((q + 1) ^ (r & 7)) << 4, c);
        }
        __syncwarp();
      }
      // the store consumed every loaded value: this warp's loads of the stage have completed
      if (lane == 0) mbar_arrive(smem_u32(&bar_rempty[s]));
      const uint32_t full = smem_u32(&bar_full[s][half]);
      advance();
      advance();
      __syncwarp();
      tmem_st_wait();
      if constexpr (kPacked) fence_proxy_async_smem();  // the tokens are read by the async proxy
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) {
          mbar_arrive(full);
        } else {
          mbar_arrive_peer(mapa_shared(full, 0));
        }
      }
      if (stages_left > 2) ok = load();
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    setmaxnreg_inc<kTmRegsEpi>();
    const int et = threadIdx.x;
    const int quad = warp & 3, half = warp >> 2, c_first = half * 32;  // every second 32-token chunk
    const int slot_row = quad * 32 + lane;                             // this thread's place in a partial's slot
    const bool storer = quad == 0 && elect_one();                      // issues its half's stores
    griddep_wait();  // xscale / xsum come from the previous kernel, and y may still be read by it
    // A thread reads the accumulator as matrix fragments: of the quadrant's lanes 8 j + lane / 4 (j < 4) the token
    // columns 2 (lane % 4) and the next of every 8.  A gated layer's lanes 0-15 hold gate rows and 16-31 the up rows of
    // the same units, so both meet in one thread.
    const int r0 = lane >> 2;
    auto row_of = [&](int tb, int j) {
      return kGated ? (2 * tb + (j >> 1)) * kBM + 64 * static_cast<int>(rank) + 16 * quad + 8 * (j & 1) + r0
                    : (2 * tb + static_cast<int>(rank)) * kBM + 32 * quad + 8 * j + r0;
    };
    // a tile's parameters, of this thread's four weight rows and, for thread et < bn, of token et; fetched a tile ahead
    float f_ws[4], f_wc[4], f_bs[4], f_xs = 0.0f;
    int f_xsum = 0;
    auto fetch = [&](int u) {
      if (u >= units) return;
      int tile, ta, tb, ka, kz;
      unit_at(u, tile, ta, tb, ka, kz);
      const int m = min(ta * bn + et, p.M - 1);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = min(row_of(tb, j), p.N - 1);
        f_ws[j] = __ldg(p.wscale + n);
        f_wc[j] = __ldg(p.wcorr + n);
        f_bs[j] = __ldg(p.bias + n);
      }
      f_xs = p.xscale[m];
      f_xsum = p.xsum[m];
    };
    fetch(unit0);
    int tile_iter = 0, chunk_iter = 0;
    for (int u = unit0; u < units; u += ustep, ++tile_iter) {
      int tile, ta, tb, ka, kz;
      unit_at(u, tile, ta, tb, ka, kz);
      const int part = u - tile * parts;
      const int buf = tile_iter & 1;
      float2 ws2[4], nwc2[4], bs2[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ws2[j] = make_float2(f_ws[j], f_ws[j]);
        nwc2[j] = make_float2(-f_wc[j], -f_wc[j]);
        bs2[j] = make_float2(f_bs[j], f_bs[j]);
      }
      tm_epi_sync();  // the previous tile's readers of the token parameters are done
      if (et < bn) {
        s_xs[et] = f_xs;
        s_cm[et] = -(8.0f * static_cast<float>(f_xsum) + p.kconst);
      }
      fetch(u + ustep);
      if (!mbar_wait(smem_u32(&bar_tfull[buf]), static_cast<uint32_t>(tile_iter >> 1) & 1u)) s_epi_abort = 1;
      tm_epi_sync();
      if (s_epi_abort) break;  // every epilogue thread leaves, or none
      tc_fence_after();
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(buf * bn);
      // r[16 g + 4 c + 2 i + k]: lane 16 g + 8 i + r0, token 8 c + 2 (lane % 4) + k of the chunk
      auto load_chunk = [&](int c0, uint32_t (&r)[32]) {
        __syncwarp();
        tmem_ld_16x256b_x4(taddr + c0, r);
        tmem_ld_16x256b_x4(taddr + (16u << 16) + c0, r + 16);
        tmem_ld_wait();
      };
      // split of K: this unit's partial to its slot; the tile's last unit adds the other units' slots to its own
      // accumulator (exact: non-negative integer multiples of one power of two, and so is their sum, below 2^24 of
      // them) and applies the epilogue.  A slot holds a thread's 32 values of each chunk as 8 float4, 128 threads apart.
      const int slot = kBM * bn / 4;
      float4* const slot4 = reinterpret_cast<float4*>(p.part_ws) + static_cast<size_t>((tile * parts + part) * 2 + static_cast<int>(rank)) * slot + slot_row;
      bool last = true;
      if (parts > 1) {
#pragma unroll 1
        for (int c0 = c_first; c0 < bn; c0 += 64) {
          uint32_t r[32];
          load_chunk(c0, r);
#pragma unroll
          for (int i = 0; i < 32; i += 4)
            __stcg(slot4 + ((c0 + i) / 4) * kBM, make_float4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]),
                                                              __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])));
        }
        tm_epi_sync();
        if (et == 0) {
          __threadfence();
          s_last = atomicAdd(p.part_cnt + tile * 2 + static_cast<int>(rank), 1) == parts - 1;
        }
        tm_epi_sync();
        last = s_last != 0;
        if (last) __threadfence();
      }
      const int m_end = min(p.M - ta * bn, bn);  // tokens of this tile
      const float2 unit2 = make_float2(262144.0f, 262144.0f);
#pragma unroll 1
      for (int c0 = c_first; c0 < m_end && last; c0 += 64, ++chunk_iter) {
        uint32_t r[32];
        load_chunk(c0, r);
#pragma unroll 1
        for (int q = 0; q < parts; ++q) {
          if (q == part) continue;
          const float4* const o4 = slot4 + static_cast<ptrdiff_t>(q - part) * 2 * slot + (c0 / 4) * kBM;
          float4 v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = __ldcg(o4 + j * kBM);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            r[4 * j] = __float_as_uint(__uint_as_float(r[4 * j]) + v[j].x);
            r[4 * j + 1] = __float_as_uint(__uint_as_float(r[4 * j + 1]) + v[j].y);
            r[4 * j + 2] = __float_as_uint(__uint_as_float(r[4 * j + 2]) + v[j].z);
            r[4 * j + 3] = __float_as_uint(__uint_as_float(r[4 * j + 3]) + v[j].w);
          }
        }
        if (p.acc != nullptr) {  // the integer accumulators, gated layers in natural order: [gate units | up units]
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int j = 2 * (i >> 4) + ((i >> 1) & 1), c = c0 + 8 * ((i >> 2) & 3) + 2 * (lane & 3) + (i & 1);
            const int n = row_of(tb, j);
            const int col = kGated ? n - (tb + (j >> 1)) * kBM + (j >> 1) * (p.N / 2) : n;
            if (n < p.N && c < m_end)
              p.acc[static_cast<size_t>(ta * bn + c) * p.N + col] =
                  static_cast<int32_t>(fmaf(__uint_as_float(r[i]), 262144.0f, s_cm[c] + nwc2[j].x));
          }
        }
        uint8_t* const out = out_smem + (2 * half + (chunk_iter & 1)) * kTmOut;
        if (storer) bulk_wait_read_but<1>();  // the store before the last has read this buffer
        tm_half_sync(half);
        uint32_t pk[4][4];  // [8-token group][row block j]: tokens 2 (lane % 4) and the next
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int t0 = c0 + 8 * c + 2 * (lane & 3);
          const float2 xs = *reinterpret_cast<const float2*>(s_xs + t0), cm = *reinterpret_cast<const float2*>(s_cm + t0);
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // exact accumulator; one float32 scale product, fma, one rounding
            const int i = 16 * (j >> 1) + 4 * c + 2 * (j & 1);
            const float2 a = __ffma2_rn(make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), unit2, __fadd2_rn(cm, nwc2[j]));
            const float2 y = __ffma2_rn(a, __fmul2_rn(xs, ws2[j]), bs2[j]);
            pk[c][j] = pack2<OutT>(y.x, y.y);
          }
        }
        // transposed 8 x 8 blocks into rows of one token (128 bytes, 128-byte swizzle: 16-byte piece q of row t at q ^ t % 8)
        if constexpr (!kGated) {  // two tiles of 64 channels; this quadrant's 32 are pieces 4 (quad % 2) .. of its tile
          const int t = lane & 7, piece = 4 * (quad & 1) + (lane >> 3);
          const uint32_t dst = smem_u32(out) + static_cast<uint32_t>((quad >> 1) * (kTmOut / 2) + t * 128 + ((piece ^ t) << 4));
#pragma unroll
          for (int c = 0; c < 4; ++c) stmatrix_x4_trans(dst + static_cast<uint32_t>(c * 1024), pk[c]);
        } else {  // one tile of 64 hidden units; this quadrant's 16 are pieces 2 quad and 2 quad + 1
          const int t = lane & 7, piece = 2 * quad + ((lane >> 3) & 1);
          const uint32_t dst = smem_u32(out) + static_cast<uint32_t>((lane >> 4) * 1024 + t * 128 + ((piece ^ t) << 4));
#pragma unroll
          for (int c = 0; c < 4; c += 2) {
            uint32_t h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              // h = gelu(gate) * up of values rounded to the output type, rounded once more
              const float2 g = unpack2<OutT>(pk[c + (i >> 1)][i & 1]), up = unpack2<OutT>(pk[c + (i >> 1)][2 + (i & 1)]);
              h[i] = pack2<OutT>(gelu_tanh(g.x) * up.x, gelu_tanh(g.y) * up.y);
            }
            stmatrix_x4_trans(dst + static_cast<uint32_t>(c * 1024), h);
          }
        }
        fence_proxy_async_smem();  // the stores are read by the async proxy
        tm_half_sync(half);
        if (storer) {  // tokens past M and channels past N are clipped
          const int m = ta * bn + c0;
          if constexpr (kGated) {
            tma_store_2d(&tmap_y, tb * kBM + 64 * static_cast<int>(rank), m, smem_u32(out));
          } else {
            const int n = (2 * tb + static_cast<int>(rank)) * kBM;
            if (n < p.N) tma_store_2d(&tmap_y, n, m, smem_u32(out));
            if (n + 64 < p.N) tma_store_2d(&tmap_y, n + 64, m, smem_u32(out + kTmOut / 2));
          }
          bulk_commit();
        }
      }
      if (parts > 1 && last && et == 0) p.part_cnt[tile * 2 + static_cast<int>(rank)] = 0;  // ready for the next launch
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) {
          mbar_arrive(smem_u32(&bar_tempty[buf]));
        } else {
          mbar_arrive_peer(mapa_shared(smem_u32(&bar_tempty[buf]), 0));
        }
      }
    }
    if (storer) bulk_wait_all();
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the leader's MMAs on this CTA's shared memory and TMEM are complete
  tc_fence_after();
  if (warp == kTmMma) tmem_dealloc_pair<512>(tmem);
}

// The layer's tiled weights, [chunks][128 rows][64 bytes], read in boxes of `rows` rows of `kbs` consecutive chunks with
// the 64-byte swizzle (16-byte piece c of row r at piece c ^ (r / 2 % 4)), which keeps the converters' 16-byte reads of
// 32 consecutive rows free of bank conflicts.
cudaError_t make_tmap_weights(CUtensorMap* m, const void* base, size_t chunks, int rows, int kbs) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {64, kBM, static_cast<cuuint64_t>(chunks)};
  const cuuint64_t strides[2] = {64, kTmRaw};
  const cuuint32_t box[3] = {64, static_cast<cuuint32_t>(rows), static_cast<cuuint32_t>(kbs)};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Packed codes [rows][width bytes], read in boxes of box_rows rows of a k-block's 64 bytes, as they are.
cudaError_t make_tmap_packed(CUtensorMap* m, const void* base, int rows, int width, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(width), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(width)};
  const cuuint32_t box[2] = {kBK / 2, static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The output [M][width] of 16-bit values, written in boxes of 64 channels x 32 tokens from 128-byte swizzled rows.
cudaError_t make_tmap_out(CUtensorMap* m, void* base, int rows, int width) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(width), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(width) * 2};
  const cuuint32_t box[2] = {64, 32};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <bool kGated, int kPlanes, bool kPacked, typename OutT>
cudaError_t launch_tm(const GemmArgs& a, int bn, int parts) {
  auto kern = gemm_tmem_kernel<kGated, kPlanes, kPacked, OutT>;
  cudaError_t e = prepare_kernel(reinterpret_cast<const void*>(kern), kTmOutBytes + kTmSmem + 1024);
  if (e != cudaSuccess) return e;
  TmParams p;
  p.xscale = a.xscale;
  p.xsum = a.xsum;
  p.wscale = a.wscale;
  p.wcorr = a.wcorr;
  p.bias = a.bias;
  p.acc = a.acc;
  p.M = a.M;
  p.N = a.N;
  p.nkb = a.K / kBK;
  p.bn = bn;
  const int btile = bn / 2 * kBK, raw = (2 / kPlanes) * kTmRaw;
  p.stages_a = (512 - 2 * bn) / (32 * (2 / kPlanes));
  if (kPacked) {  // the expanded tokens are as deep as the weight stages, the packed codes as the packed weights
    while ((p.stages = (kTmSmem - p.stages_a * 2 * btile) / (raw + btile)) < p.stages_a + 2) --p.stages_a;
  } else {
    p.stages = kTmSmem / (2 * btile + raw);
  }
  if (p.stages > kTmMaxStages) p.stages = kTmMaxStages;
  if (p.stages_a > p.stages - 2) p.stages_a = p.stages - 2;
  p.tiles_m = (a.M + bn - 1) / bn;
  p.tiles_n = (a.N + 255) / 256;
  p.parts = parts;
  p.part_ws = a.part_ws;
  p.part_cnt = a.part_cnt;
  p.kconst = (kPlanes == 2 ? 1024.0f : 64.0f) * static_cast<float>(a.K);
  CUtensorMap tx = {}, tw = {}, ty = {};
  e = kPacked ? make_tmap_packed(&tx, a.xq, a.M, a.K / 2, bn / 2) : make_tmap_bytes(&tx, a.xq, a.M, kPlanes * a.K, bn / 2);
  if (e == cudaSuccess) e = make_tmap_weights(&tw, a.wq, static_cast<size_t>(p.tiles_n) * 2 * p.nkb, kGated ? 64 : 128, 2 / kPlanes);
  if (e == cudaSuccess) e = make_tmap_out(&ty, a.y, a.M, a.gated ? a.N / 2 : a.N);
  if (e != cudaSuccess) return e;
  const int units = p.tiles_m * p.tiles_n * parts, pairs = a.num_sms / 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * (units < pairs ? units : pairs)));
  cfg.blockDim = dim3(kTmThreads);
  cfg.dynamicSmemBytes = kTmOutBytes + kTmSmem + 1024;
  cfg.stream = a.stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, kern, tx, tw, ty, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// Estimated time (ns) of a launch with tiles of bn tokens in `parts` work units, fitted to GB300 measurements (1876 launches,
// M 5-1500, K 128-16384, weight rows 16-32768: within 16%, half of them within 4%): a fixed cost, more with more pairs at
// work, with the last tile's epilogue; the first unit's k-blocks (165 ns each up to bn = 128, 172 at 160, 200 at 192; two
// planes 250, or 1.95 bn; packed codes 235 to 290); per further wave of pairs a unit's k-blocks and hand-over, or the epilogue where that is
// longer; with K split, the partial's write and read-back.
long tm_estimate(const GemmArgs& a, int bn, int parts) {
  const long pairs = a.num_sms / 2, nkb = a.K / kBK;
  const long units = static_cast<long>((a.M + bn - 1) / bn) * ((a.N + 255) / 256) * parts;
  const long waves = (units + pairs - 1) / pairs;
  const long kb = a.x_bytes == 2   ? (bn <= 128 ? 250 : 195l * bn / 100)
                  : a.x_bytes == 0 ? (bn <= 64 ? 235 : bn <= 96 ? 264 : bn <= 128 ? 270 : bn <= 160 ? 285 : 290)
                                   : (bn <= 128 ? 165 : bn <= 160 ? 172 : 200);
  const long work = (nkb + parts - 1) / parts * kb;
  const long split = parts > 1 ? 1500 + 7l * parts * bn : 0;
  long unit = work + (bn > 160 ? 580 : 870) + (a.gated ? 150 : 0);
  const long epilogue = a.gated ? 1000 + 19l * bn / 2 : 800 + 17l * bn / 2;
  if (unit < epilogue) unit = epilogue;
  return 3000 + 28 * (units < pairs ? units : pairs) + 8l * bn + (a.gated ? 200 : 0) + work + split + (waves - 1) * (unit + split);
}

template <int kPlanes, bool kPacked, typename OutT>
cudaError_t launch_tm_g(const GemmArgs& a, int bn, int parts) {
  return a.gated ? launch_tm<true, kPlanes, kPacked, OutT>(a, bn, parts) : launch_tm<false, kPlanes, kPacked, OutT>(a, bn, parts);
}

}  // namespace

// A split needs the workspace's room, units of at least 8 k-blocks, and an estimate 10% below whole tiles.
long gemm_tmem_plan(const GemmArgs& a, int* bn, int* parts) {
  const bool can_split = !a.gated && a.x_bytes == 1 && a.part_ws != nullptr && a.part_cnt != nullptr;
  const long nkb = a.K / kBK, tiles_n = (a.N + 255) / 256;
  long best = -1;
  for (int w = kTmMaxBn; w >= 32; w -= 32) {
    const long t = tm_estimate(a, w, 1);
    if (best < 0 || t < best) {
      best = t;
      *bn = w;
      *parts = 1;
    }
  }
  const long whole = best;
  for (int w = kTmMaxBn; can_split && w >= 32; w -= 32) {
    const long tiles = (a.M + w - 1) / w * tiles_n;
    for (int q = 2; q <= 4; q *= 2) {
      if (nkb / q < 8 || static_cast<size_t>(tiles) * q * 2 * kBM * w > a.part_ws_floats || 2 * tiles > a.part_cnt_n) continue;
      const long t = tm_estimate(a, w, q);
      if (t < best && 10 * t < 9 * whole) {
        best = t;
        *bn = w;
        *parts = q;
      }
    }
  }
  return best;
}

cudaError_t launch_gemm_tmem(const GemmArgs& a, int bn, int parts) {
  if (a.x_bytes == 2)
    return a.ydt == 0 ? launch_tm_g<2, false, __half>(a, bn, parts) : launch_tm_g<2, false, __nv_bfloat16>(a, bn, parts);
  if (a.x_bytes == 0)
    return a.ydt == 0 ? launch_tm_g<1, true, __half>(a, bn, parts) : launch_tm_g<1, true, __nv_bfloat16>(a, bn, parts);
  return a.ydt == 0 ? launch_tm_g<1, false, __half>(a, bn, parts) : launch_tm_g<1, false, __nv_bfloat16>(a, bn, parts);
}

cudaError_t read_and_clear_error_word_tmem(unsigned int* out, cudaStream_t stream) {
  cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyFromSymbol(out, g_error_word, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  const unsigned int zero = 0;
  return cudaMemcpyToSymbol(g_error_word, &zero, sizeof(unsigned int));
}

cudaError_t set_debug_hooks_tmem(unsigned long long wait_limit_ns, int hold_loads) {
  return set_debug_hooks(wait_limit_ns, hold_loads);
}

}  // namespace qvla
