// W4A8 variant of the integer GEMM: int8 activation codes against int4 weight codes that carry one
// fp32 scale per (output channel, 128 consecutive k):
//     y[m, n] = sx[m] * sum_kg sw4[n, kg] * ( sum_{k in kg} q[m, k] * q4[n, k] ) + bias[n]
//
// The product is formed TRANSPOSED: the weights are the M operand of the tensor core (128 output channels = the 128
// lanes of tensor memory) and the activation codes the N operand (128 tokens = columns).  A drain thread then owns ONE
// output channel for 64 tokens, so the group's scale is one register per k-block instead of a table look-up per column.
//
// The k-block of the pipeline is exactly one scale group.  Per k-block:
//   warp 0       TMA of the 128 x 128-byte tile of activation codes
//   warp 1       four tcgen05.mma kind::i8 (128 x 128 x 32) into a FRESH accumulator of 128 tensor-memory columns; two
//                k-blocks are handed to the drain at a time
//   warps 2-7    two warps per k-block, three k-blocks in turn: TMA of the packed nibbles of 64 channels (weights are
//                constants: the first tiles are requested before the kernel that produces the codes has finished),
//                unpacked in registers: 16 bytes of nibbles -> 32 int8 (nibble << 4, i.e. 16 * q4, which is sign-correct
//                without any sign extension) written in the 128-byte-swizzled K-major layout the tensor core reads
//   warps 8-15   drain: S[m] += acc[m] * mult[kg][n].  mult are the group scales of a channel on a common power-of-two
//                grid (sw4[n,kg] = mult[kg][n] * base[n]), so the sum over groups is EXACT integer arithmetic and no
//                cancellation between groups can lose bits.
// At the end of a tile the sums are converted once: y = fma(float(S), sx * base[n], bias[n]),
// with the same cancellation check against the bias as the 8-bit kernel, transposed through a staging tile in shared
// memory and written by TMA stores.  Every wait is bounded.
//
// The drain holds S, up to 2^50, as two 32-bit numbers instead of multiplying 32 x 32 -> 64 bits:
//   L = S mod 2^32          (one 32-bit multiply-add)
//   F = S within 2^31       (one conversion and one fp32 FMA; F moves in one binade, so that every addition rounds to a multiple of 2^kGrid)
// and S = f 2^kGrid + D with f the steps that F has moved and D the signed 32-bit remainder of L: as exact as the 64-bit sum.  An addition
// rounds F by half a step at most, so |D| <= 9 * 2^27 < 2^31 after nine k-blocks.  S stays within 2^50 for mult below 2^b,
// b = 33 - ceil(log2(14 K / 128)): 26 bits at K = 1152.  A channel whose scales need more (exponents that span more than three binades; a ratio
// below four never does) is marked by the sign of base, and a warp that holds one adds 64-bit products with all 30 bits of mult.  Longer
// reductions do so throughout: with 25 bits few channels qualify, and of the 32 of a warp hardly ever all.  So do small problems (see launch_gemm_w4).
//
// What bounds it: the drain.  Clocks per k-block of 128 x 128 accumulators for the drain loop by itself: 64-bit multiply-adds 603, L and F 453, one
// fp32 conversion and FMA 322, the loads from tensor memory 185; 256 of tensor pipe.  In the kernel a k-block takes about 1000, and a tile
// 4000 more for conversion and output.  M = 16384, microseconds with 64-bit sums throughout -> now:
// 1152 -> 4608 221 -> 203 (with GELU 260 -> 243), 1152 -> 3456 168 -> 155; 4608 -> 1152 170
// either way; the layers alternating in a block together 738 -> 730.
// Measured and not better: a CTA pair sharing the codes and sixteen drain warps of 32 tokens (64-bit sums: 1152 -> 4608 221 -> 211 and 218, 1152 -> 1152
// 59 -> 64 and 58); sums in fp64 (260 -> 358); weights unpacked into tensor memory with the codes of a token tile resident and one k-block
// per hand-over (221 -> 238, 4608 -> 1152 170 -> 180: four unpack warps and one instruction cache for everything); nibbles unpacked to q4 instead of
// 16 q4, which would give b four more bits (four more instructions per eight weights: 4608 -> 1152 170 -> 190).
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace trdq {
namespace {

constexpr int kTileTok = 128;    // tokens per tile: N of the MMA
constexpr int kTileCh = 128;     // output channels per tile: M of the MMA, lanes of tensor memory
constexpr int kTileK = 128;
constexpr int kUnpackWarps = 6;
constexpr int kUnpackSplit = 2;    // warps that share a k-block
constexpr int kUnpackTurns = kUnpackWarps / kUnpackSplit;
constexpr int kDrainWarps = 8;   // 4 lane quarters x 2 groups of 64 tokens
constexpr int kThreads = 32 * (2 + kUnpackWarps + kDrainWarps);
constexpr int kTokPerWarp = kTileTok / (kDrainWarps / 4);
constexpr int kHandoff = 2;      // k-blocks per hand-over to the drain
constexpr int kSlots = 2;        // hand-overs in flight: kSlots * kHandoff accumulators of 128 columns
constexpr int kTmemCols = 512;
constexpr int kW8Bytes = kTileCh * kTileK;         // 16 KB int8 weights after unpacking
constexpr int kTokBytes = kTileTok * kTileK;       // 16 KB activation codes
constexpr int kStageBytes = kW8Bytes + kTokBytes;
constexpr int kStages = 4;
constexpr int kPackedBytes = kTileCh / kUnpackSplit * 64;  // 4 KB nibbles of one unpack warp
constexpr int kPackedDepth = 2;                    // packed tiles in flight per unpack warp
constexpr int kPackedStages = kPackedDepth * kUnpackWarps;
constexpr int kOutStageBytes = kDrainWarps * kTokPerWarp * 64;  // per drain warp 64 tokens x 32 channels bf16
constexpr int kSxBytes = kDrainWarps * kTokPerWarp * 4;
constexpr int kBarrierBytes = 512;
constexpr int kPackedOff = kStages * kStageBytes;
constexpr int kOutOff = kPackedOff + kPackedStages * kPackedBytes;
constexpr int kSxOff = kOutOff + kOutStageBytes;
constexpr int kBarOff = kSxOff + kSxBytes;
constexpr int kSmemBytes = 1024 + kBarOff + kBarrierBytes;
static_assert(kSmemBytes <= 227 * 1024, "shared memory");
static_assert(kSlots * kHandoff * kTileTok <= kTmemCols, "tensor memory");
// Registers: 512 threads are launched with 128 each.  The two drain warpgroups need the 128 of their 64-bit sums plus a
// double-buffered tensor-memory load, the other two few: 128 * (2 * 192 + 2 * 64) = the 512 * 128 of the launch.
constexpr int kRegsLaunch = 128, kRegsDrain = 192, kRegsOther = 64;
static_assert(kDrainWarps * 32 * kRegsDrain + (kThreads - kDrainWarps * 32) * kRegsOther <= kThreads * kRegsLaunch, "register split exceeds the launch's allocation");

// The drain's numbers: mult has kMultBits bits, a step of F is 2^kGrid.
constexpr int kMultBits = 30, kGrid = 28, kMinFastBits = 26;
constexpr float kAnchor = 3377699720527872.0f;  // 1.5 * 2^51: one binade for sums within +- 2^50, its float steps are 2^28
constexpr uint32_t kAnchorBits = 0x59400000u;
constexpr int64_t kFastBlocksPerSm = 200;
// bits of mult with which sums of `groups` k-blocks stay within +- 2^50: |acc| <= 16 * 128 * 7 * 128 = 14 * 2^17
__host__ __device__ constexpr int w4_fast_bits(int groups) {
  int log = 0;
  while (static_cast<int64_t>(1) << log < static_cast<int64_t>(14) * groups) ++log;
  return 33 - log < kMultBits ? 33 - log : kMultBits;
}
// kMinFastBits: at most nine additions, so the remainder stays below 9 * 2^(kGrid - 1)
static_assert(w4_fast_bits(9) >= kMinFastBits && w4_fast_bits(10) < kMinFastBits && 9 < (1 << (32 - kGrid)), "the remainder has to fit 32 signed bits");

struct alignas(64) W4Params {
  CUtensorMap tmap_a[2];    // codes of each segment, box 128 B x 128 rows, 128-byte swizzle
  CUtensorMap tmap_b;       // packed weights, box 64 B x 64 rows
  CUtensorMap tmap_out[2];  // bf16 output, box 32 channels x 64 tokens, 64-byte swizzle
  const float* sx[2];
  int32_t M[2];
  int32_t tiles_m[2];
  const int32_t* mult_t;  // [K/128][n_pad]
  const float* base;      // [n_pad], negative: the channel needs more than w4_fast_bits
  const __nv_bfloat16* bias;
  int32_t N, K, tiles_n, n_pad;
  int32_t fast_shift;     // kMultBits - w4_fast_bits
  uint32_t* status;
};

struct TileCoord {
  int seg, m0, n0;
};
__device__ __forceinline__ TileCoord tile_coord(const W4Params& p, int tile) {
  const int tiles_m = p.tiles_m[0] + p.tiles_m[1];
  const int nt = tile / tiles_m;
  int mt = tile - nt * tiles_m;
  TileCoord c;
  c.seg = mt >= p.tiles_m[0] ? 1 : 0;
  if (c.seg) mt -= p.tiles_m[0];
  c.m0 = mt * kTileTok;
  c.n0 = nt * kTileCh;
  return c;
}

struct Ring {
  int idx = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void advance(int n) {
    if (++idx == n) {
      idx = 0;
      phase ^= 1;
    }
  }
};

// Waits for this thread's tensor-memory loads; every use of the registers stays behind the wait.
__device__ __forceinline__ void tmem_wait_ld_regs(uint32_t (&r)[16]) {
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
}

// What a drain thread adds up for its channel, a sum for each of its tokens.
template <bool WIDE>
struct ChannelSums;
template <>
struct ChannelSums<false> {
  uint32_t L[kTokPerWarp];
  float F[kTokPerWarp];
  uint32_t mult;
  float multf;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < kTokPerWarp; ++j) {
      L[j] = 0;
      F[j] = kAnchor;
    }
  }
  __device__ __forceinline__ void set_mult(int32_t m, int shift) {
    mult = static_cast<uint32_t>(m >> shift);
    multf = __int2float_rn(m >> shift);  // exact: 24 significant bits
  }
  __device__ __forceinline__ void add(int j, uint32_t acc) {
    L[j] += acc * mult;
    F[j] = __fmaf_rn(__int2float_rn(static_cast<int32_t>(acc)), multf, F[j]);
  }
  __device__ __forceinline__ int32_t rest(int j) const {  // (the anchor's low bits are zero)
    return static_cast<int32_t>(L[j] - (__float_as_uint(F[j]) << kGrid));
  }
  __device__ __forceinline__ long long whole(int j) const {
    return (static_cast<long long>(static_cast<int32_t>(__float_as_uint(F[j]) - kAnchorBits)) << kGrid) + rest(j);
  }
  // eight sums as floats
  __device__ __forceinline__ void to_float(int j0, float (&v)[8]) const {
    float low = __uint_as_float(0x7F800000u);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      v[e] = __fadd_rn(__fsub_rn(F[j0 + e], kAnchor), __int2float_rn(rest(j0 + e)));
      if (e & 1) low = min3_abs(low, v[e - 1], v[e]);
    }
    if (low < 1073741824.0f) {  // below 2^30 the sum is L itself: no rounding of the remainder on the way
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (fabsf(v[e]) < 1073741824.0f) v[e] = __int2float_rn(static_cast<int32_t>(L[j0 + e]));
    }
  }
};
template <>
struct ChannelSums<true> {
  long long sum[kTokPerWarp];
  int32_t mult;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < kTokPerWarp; ++j) sum[j] = 0;
  }
  __device__ __forceinline__ void set_mult(int32_t m, int) {
    mult = m;
    asm volatile("" : "+r"(mult));  // stays a 32-bit factor: widened ahead of the loop it would cost a 64 x 64 product
  }
  __device__ __forceinline__ void add(int j, uint32_t acc) {
    sum[j] += static_cast<long long>(static_cast<int32_t>(acc)) * static_cast<long long>(mult);
  }
  __device__ __forceinline__ long long whole(int j) const { return sum[j]; }
  __device__ __forceinline__ void to_float(int j0, float (&v)[8]) const {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __ll2float_rn(sum[j0 + e]);
  }
};

// State of a drain warp that lasts from tile to tile.
struct DrainState {
  BoundedWaiter w;
  Ring slot;
  uint32_t bar_full, bar_empty;  // of the hand-overs
  uint32_t t_lane;               // tensor-memory address of this warp's lanes and first token
  uint32_t stage;                // its staging tile
  float* sx;                     // the row scales of its tokens
  int lane;
  int32_t m_next;                // multiplier of the next k-block
};

// One tile of one drain warp: sums over the k-blocks, then y = float(S) * (sx * base) + bias (base is a power of two: the product is
// exact) into the staging tile.  `next`: first multiplier of the warp's next tile.
// WIDE: a channel of the warp needs all bits of mult.  ACT: GELU (tanh form) on the dequantized value before the bf16 rounding.
template <bool WIDE, bool ACT>
__device__ __forceinline__ void drain_tile(const W4Params& p, DrainState& s, int n, float base, float bias, int num_kb, const int32_t* next,
                                           const float (&sx_reg)[kTokPerWarp / 32]) {
  ChannelSums<WIDE> acc;
  acc.clear();
  const int shift = WIDE ? 0 : p.fast_shift;
  const int32_t* mp = p.mult_t + n;
  // Two register buffers: a tensor-memory load is always in flight behind the multiply-adds, across k-blocks too.
  uint32_t r[2][16];
  s.w.wait(s.bar_full + 8 * s.slot.idx, s.slot.phase);
  __syncwarp();
  tc_fence_after();
  uint32_t t_row = s.t_lane + s.slot.idx * (kHandoff * kTileTok);
  tmem_ld_32x16(t_row, r[0]);
#pragma unroll 1
  for (int kb = 0; kb < num_kb; ++kb) {
    acc.set_mult(s.m_next, shift);
    if (kb + 1 < num_kb) {
      mp += p.n_pad;
      s.m_next = __ldg(mp);
    }
    const bool hand_back = kb % kHandoff == kHandoff - 1 || kb + 1 == num_kb;
#pragma unroll
    for (int ch = 0; ch < kTokPerWarp / 16; ++ch) {
      tmem_wait_ld_regs(r[ch & 1]);
      if (ch + 1 < kTokPerWarp / 16) {
        tmem_ld_32x16(t_row + (ch + 1) * 16, r[(ch + 1) & 1]);
      } else if (!hand_back) {
        t_row += kTileTok;
        tmem_ld_32x16(t_row, r[0]);
      } else {
        tc_fence_before();
        __syncwarp();
        if (s.lane == 0) mbar_arrive(s.bar_empty + 8 * s.slot.idx);
        s.slot.advance(kSlots);
        if (kb + 1 < num_kb) {
          s.w.wait(s.bar_full + 8 * s.slot.idx, s.slot.phase);
          __syncwarp();
          tc_fence_after();
          t_row = s.t_lane + s.slot.idx * (kHandoff * kTileTok);
          tmem_ld_32x16(t_row, r[0]);
        }
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) acc.add(ch * 16 + j, r[ch & 1][j]);
    }
  }

  if (next) s.m_next = __ldg(next);
  const float unit = __fmul_rn(base, static_cast<float>(1 << shift));
  const float thr = fabsf(bias) * 0.0009765625f;
  // byte of this lane's channel inside a staging row (64 bytes, 64-byte swizzle: 16-byte chunk index xor row bits 1..2)
  const uint32_t lane_chunk = s.lane >> 3, lane_byte = (s.lane & 7) * 2;
  if (s.lane == 0) bulk_wait_group_read<0>();  // the previous store has finished reading the staging tile
#pragma unroll
  for (int i = 0; i < kTokPerWarp / 32; ++i) s.sx[32 * i + s.lane] = sx_reg[i];
  __syncwarp();
  // Eight tokens at a time without a branch between them (a branch per value serialises conversion, product and
  // store); the rare cancellation against the bias is repaired for the whole group.
#pragma unroll
  for (int j0 = 0; j0 < kTokPerWarp; j0 += 8) {
    float v[8], y[8];
    acc.to_float(j0, v);
    const float4 sa = *reinterpret_cast<const float4*>(s.sx + j0), sb = *reinterpret_cast<const float4*>(s.sx + j0 + 4);
    const float sx8[8] = {sa.x, sa.y, sa.z, sa.w, sb.x, sb.y, sb.z, sb.w};
    bool cancels = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      y[e] = __fmaf_rn(v[e], __fmul_rn(sx8[e], unit), bias);
      cancels |= fabsf(y[e]) < thr;
    }
    if (cancels) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        // the part of the sum that fp32 dropped
        if (fabsf(y[e]) < thr) y[e] = __fmaf_rn(__ll2float_rn(acc.whole(j0 + e) - __float2ll_rz(v[e])), __fmul_rn(sx8[e], unit), y[e]);
      }
    }
    uint32_t packed[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float2 two = make_float2(y[2 * g], y[2 * g + 1]);
      packed[g] = pack_bf16(ACT ? gelu_tanh2<false>(two) : two);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int j = j0 + e;
      const uint16_t h = static_cast<uint16_t>(packed[e / 2] >> (16 * (e & 1)));
      asm volatile("st.shared.u16 [%0], %1;" ::"r"(s.stage + j * 64 + ((lane_chunk ^ ((j >> 1) & 3)) << 4) + lane_byte), "h"(h) : "memory");
    }
  }
}

// ACT: GELU (tanh form) on the dequantized value before the bf16 rounding.  FAST: reductions of up to nine k-blocks, with both forms of the
// sum; longer ones have a kernel with the 64-bit form alone, which is half the instructions (40 KB against 73, with GELU 53 against 98).
template <bool ACT, bool FAST>
__global__ void __launch_bounds__(kThreads, 1) gemm_w4a8_kernel(const __grid_constant__ W4Params p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kBarOff);
  const uint32_t bar_full = smem_u32(bars);                // [kStages]        codes landed and weights unpacked
  const uint32_t bar_empty = bar_full + 8 * kStages;       // [kStages]        the MMAs have read the stage
  const uint32_t bar_praw = bar_empty + 8 * kStages;       // [kPackedStages]  nibbles landed
  const uint32_t bar_tfull = bar_praw + 8 * kPackedStages; // [kSlots]         accumulators complete
  const uint32_t bar_tempty = bar_tfull + 8 * kSlots;      // [kSlots]         accumulators drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + kPackedStages + 2 * kSlots);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int total_tiles = (p.tiles_m[0] + p.tiles_m[1]) * p.tiles_n;
  const int num_kb = p.K / kTileK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar_full + 8 * s, 1 + kUnpackSplit);  // one arrive.expect_tx for the codes, the unpack warps
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int s = 0; s < kPackedStages; ++s) mbar_init(bar_praw + 8 * s, 1);
    for (int a = 0; a < kSlots; ++a) {
      mbar_init(bar_tfull + 8 * a, 1);
      mbar_init(bar_tempty + 8 * a, kDrainWarps);
    }
    fence_mbar_init();
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  griddep_launch_dependents();
  const int my_tiles = static_cast<int>(blockIdx.x) < total_tiles ? (total_tiles - 1 - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x) + 1 : 0;
  const int total_kb = my_tiles * num_kb;

  if (warp >= kThreads / 32 - kDrainWarps) {
    // ------------------------------------------------------------------- drain
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsDrain));
    griddep_wait();
    const int dw = warp - (kThreads / 32 - kDrainWarps);
    const int q = dw & 3;           // = warp % 4: the lane quarter of tensor memory this warp may read
    const int tok_off = (dw >> 2) * kTokPerWarp;
    const uint32_t my_stage = smem_base + kOutOff + dw * (kTokPerWarp * 64);
    float* my_sx = reinterpret_cast<float*>(smem + kSxOff) + dw * kTokPerWarp;
    const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + tok_off;
    const int lane_n = q * 32 + lane;
    DrainState s{BoundedWaiter(p.status, kStatusTimeoutEpilogue), Ring(), bar_tfull, bar_tempty, t_lane, my_stage, my_sx, lane,
                 my_tiles > 0 ? __ldg(p.mult_t + tile_coord(p, blockIdx.x).n0 + lane_n) : 0};
    for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
      const TileCoord tc = tile_coord(p, tile);
      const int n = tc.n0 + lane_n;  // < n_pad
      // requested here, used after the last k-block: an L2 round trip is about as long as a k-block
      const float base = __ldg(p.base + n);
      const uint16_t bias_bits = p.bias && n < p.N ? __ldg(reinterpret_cast<const uint16_t*>(p.bias) + n) : 0;
      const float bias = __uint_as_float(static_cast<uint32_t>(bias_bits) << 16);
      float sx_reg[kTokPerWarp / 32];
#pragma unroll
      for (int i = 0; i < kTokPerWarp / 32; ++i) {
        const int row = tc.m0 + tok_off + 32 * i + lane;
        sx_reg[i] = row < p.M[tc.seg] ? __ldg(p.sx[tc.seg] + row) : 0.0f;
      }
      const int after = tile + static_cast<int>(gridDim.x);
      const int32_t* next = after < total_tiles ? p.mult_t + tile_coord(p, after).n0 + lane_n : nullptr;
      if (!FAST || __any_sync(0xffffffffu, base < 0.0f)) {
        drain_tile<true, ACT>(p, s, n, fabsf(base), bias, num_kb, next, sx_reg);
      } else if constexpr (FAST) {
        drain_tile<false, ACT>(p, s, n, base, bias, num_kb, next, sx_reg);
      }
      fence_proxy_async_smem();
      __syncwarp();  // (the reads of my_sx are done as well)
      if (lane == 0) {
        tma_store_2d(&p.tmap_out[tc.seg], tc.n0 + q * 32, tc.m0 + tok_off, my_stage);  // rows >= M and columns >= N are clipped
        bulk_commit_group();
      }
    }
    if (lane == 0) bulk_wait_group_read<0>();  // the staging tiles have been read; the stores complete before the grid does
    s.w.settle();
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == 0) {
      // ------------------------------------------------- TMA of the activation codes
      if (elect_one()) {
        prefetch_tensormap(&p.tmap_a[0]);
        prefetch_tensormap(&p.tmap_a[1]);
        prefetch_tensormap(&p.tmap_out[0]);
        prefetch_tensormap(&p.tmap_out[1]);
        griddep_wait();  // the codes come from the kernel before
        BoundedWaiter w(p.status, kStatusTimeoutProducer);
        Ring st;
        for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
          const TileCoord tc = tile_coord(p, tile);
          for (int kb = 0; kb < num_kb; ++kb) {
            w.wait(bar_empty + 8 * st.idx, st.phase ^ 1);
            mbar_arrive_expect_tx(bar_full + 8 * st.idx, kTokBytes);
            tma_load_2d(smem_base + st.idx * kStageBytes + kW8Bytes, &p.tmap_a[tc.seg], kb * kTileK, tc.m0, bar_full + 8 * st.idx);
            st.advance(kStages);
          }
        }
        w.settle();
      }
    } else if (warp == 1) {
      // ------------------------------------------------- MMA issuer
      if (elect_one()) {
        BoundedWaiter w(p.status, kStatusTimeoutMma);
        constexpr uint32_t idesc = umma_idesc_s8(kTileTok);
        Ring st, slot;
        for (int t = 0; t < my_tiles; ++t) {
          for (int kb = 0; kb < num_kb; ++kb) {
            const int h = kb % kHandoff;
            if (h == 0) w.wait(bar_tempty + 8 * slot.idx, slot.phase ^ 1);  // accumulators drained
            w.wait(bar_full + 8 * st.idx, st.phase);                        // codes landed, weights unpacked
            tc_fence_after();
            const uint32_t w_addr = smem_base + st.idx * kStageBytes;
            const uint64_t a_desc = umma_desc_k_sw128(w_addr);
            const uint64_t b_desc = umma_desc_k_sw128(w_addr + kW8Bytes);
            const uint32_t d_tmem = tmem_base + (slot.idx * kHandoff + h) * kTileTok;
#pragma unroll
            for (int k = 0; k < kTileK / 32; ++k) umma_i8(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, k != 0 ? 1u : 0u);
            umma_commit(bar_empty + 8 * st.idx);
            st.advance(kStages);
            if (h == kHandoff - 1 || kb + 1 == num_kb) {
              umma_commit(bar_tfull + 8 * slot.idx);
              slot.advance(kSlots);
            }
          }
        }
        w.settle();
      }
    } else {
      // ------------------------------------------------- unpack nibbles -> int8, k-blocks i = turn (mod 3), 64 of the tile's channels
      // The nibbles are requested without waiting for the kernel before: the weights are constants of the prepared
      // object, and the last kernel of their preparation (w4_multipliers_kernel, an ordinary launch) is complete before
      // this kernel's predecessor can start.
      const int uw = warp - 2;
      const int turn = uw / kUnpackSplit, part = uw % kUnpackSplit;
      BoundedWaiter w(p.status, kStatusTimeoutUnpack);
      const uint32_t my_packed = smem_base + kPackedOff + uw * kPackedDepth * kPackedBytes;
      const uint32_t my_praw = bar_praw + 8 * uw * kPackedDepth;
      auto request = [&](int i, int slot_idx) {  // lane 0: the nibbles of this CTA's k-block i
        const int t = i / num_kb;
        const TileCoord tc = tile_coord(p, blockIdx.x + t * gridDim.x);
        mbar_arrive_expect_tx(my_praw + 8 * slot_idx, kPackedBytes);
        tma_load_2d(my_packed + slot_idx * kPackedBytes, &p.tmap_b, (i - t * num_kb) * (kTileK / 2), tc.n0 + part * (kTileCh / kUnpackSplit), my_praw + 8 * slot_idx);
      };
      if (lane == 0) {
        prefetch_tensormap(&p.tmap_b);
        for (int d = 0; d < kPackedDepth; ++d)
          if (turn + d * kUnpackTurns < total_kb) request(turn + d * kUnpackTurns, d);
      }
      __syncwarp();
      Ring ps;
      for (int i = turn; i < total_kb; i += kUnpackTurns) {
        w.wait(my_praw + 8 * ps.idx, ps.phase);
        const int st_idx = i % kStages;
        w.wait(bar_empty + 8 * st_idx, ((i / kStages) & 1) ^ 1);
        __syncwarp();
        const uint32_t bp = my_packed + ps.idx * kPackedBytes;
        const uint32_t w8 = smem_base + st_idx * kStageBytes + part * (kW8Bytes / kUnpackSplit);
#pragma unroll 1
        for (int c = 0; c < 4 / kUnpackSplit; ++c) {
          // 16-byte source chunks: channel = id / 4, chunk = id % 4, id = lane + 32 (4 c + i); four in flight at once
          uint4 src[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(src[k].x), "=r"(src[k].y), "=r"(src[k].z), "=r"(src[k].w)
                         : "r"(bp + (lane + 32 * (4 * c + k)) * 16)
                         : "memory");
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int id = lane + 32 * (4 * c + k);
            const int row = id >> 2, sc = id & 3;
            const uint32_t wsrc[4] = {src[k].x, src[k].y, src[k].z, src[k].w};
            uint32_t o[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t even = (wsrc[j] << 4) & 0xF0F0F0F0u;  // k even: low nibble moved to the high half
              const uint32_t odd = wsrc[j] & 0xF0F0F0F0u;          // k odd: already in the high half
              o[2 * j] = __byte_perm(even, odd, 0x5140);
              o[2 * j + 1] = __byte_perm(even, odd, 0x7362);
            }
            const uint32_t dst_row = w8 + row * 128;
            st_shared_v4(dst_row + (((2 * sc) ^ (row & 7)) << 4), o[0], o[1], o[2], o[3]);
            st_shared_v4(dst_row + (((2 * sc + 1) ^ (row & 7)) << 4), o[4], o[5], o[6], o[7]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar_full + 8 * st_idx);
          if (i + kPackedDepth * kUnpackTurns < total_kb) request(i + kPackedDepth * kUnpackTurns, ps.idx);
        }
        ps.advance(kPackedDepth);
      }
      w.settle();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// One thread per output channel (and time-step group, blockIdx.y): put the channel's group scales on a common power-of-two grid.
__global__ void w4_multipliers_kernel(const float* __restrict__ scales, int32_t N, int32_t groups, int32_t n_pad,
                                      int32_t* __restrict__ mult_t, float* __restrict__ base) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= n_pad) return;
  scales += static_cast<int64_t>(blockIdx.y) * N * groups;
  mult_t += static_cast<int64_t>(blockIdx.y) * groups * n_pad;
  base += static_cast<int64_t>(blockIdx.y) * n_pad;
  if (n >= N) {
    for (int g = 0; g < groups; ++g) mult_t[static_cast<int64_t>(g) * n_pad + n] = 0;
    base[n] = 0.0f;
    return;
  }
  float smax = 0.0f;
  for (int g = 0; g < groups; ++g) smax = fmaxf(smax, scales[static_cast<int64_t>(n) * groups + g]);
  int e_max = 0;
  frexpf(smax, &e_max);  // smax = f * 2^e_max, f in [0.5, 1); smax == 0 gives e_max = 0
  if (e_max < -90) e_max = -90;  // keeps base a normal number; such channels are numerically zero anyway
  int32_t all = 0;
  for (int g = 0; g < groups; ++g) {
    const float s = scales[static_cast<int64_t>(n) * groups + g];
    const int32_t m = __float2int_rn(ldexpf(s, kMultBits - e_max));  // < 2^30, exact if the exponents span < 7 bits
    mult_t[static_cast<int64_t>(g) * n_pad + n] = m;
    all |= m;
  }
  // (a scale that is not a finite number gives a mult past 2^30)
  const bool wide = w4_fast_bits(groups) < kMinFastBits || (all >> kMultBits) != 0 || (all & ((1 << (kMultBits - w4_fast_bits(groups))) - 1)) != 0;
  // the tensor core sees 16 * q4 (the nibble sits in the high half of the byte): fold the 1/16 here
  const float unit = ldexpf(1.0f, e_max - kMultBits - 4);
  base[n] = wide ? -unit : unit;
}

}  // namespace

cudaError_t launch_w4_multipliers(const float* scales, int32_t N, int32_t groups, int32_t n_pad, int sets, int32_t* mult_t, float* base,
                                  cudaStream_t stream) {
  constexpr int kMaxGridY = 65535;
  for (int first = 0; first < sets; first += kMaxGridY) {
    const int count = sets - first < kMaxGridY ? sets - first : kMaxGridY;
    w4_multipliers_kernel<<<dim3((n_pad + 127) / 128, count), 128, 0, stream>>>(
        scales + static_cast<int64_t>(first) * N * groups, N, groups, n_pad, mult_t + static_cast<int64_t>(first) * groups * n_pad,
        base + static_cast<int64_t>(first) * n_pad);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

trdq_status launch_gemm_w4(const trdq_weights* w, int g, const GemmSegment seg[2], const void* bias_bf16, cudaStream_t stream, int act) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) != cudaSuccess) return TRDQ_ERR_CUDA;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  W4Params p;
  int64_t tiles_m = 0;
  for (int s = 0; s < 2; ++s) {
    p.sx[s] = seg[s].sx;
    p.M[s] = seg[s].M;
    p.tiles_m[s] = (seg[s].M + kTileTok - 1) / kTileTok;
    tiles_m += p.tiles_m[s];
  }
  if (tiles_m == 0) return TRDQ_OK;
  for (int s = 0; s < 2; ++s) {
    if (seg[s].M == 0) continue;
    const GemmSegment& src = seg[s];
    trdq_status st = encode_tmap_u8_sw128(&p.tmap_a[s], src.codes, static_cast<uint64_t>(w->K), static_cast<uint64_t>(src.M),
                                          static_cast<uint64_t>(w->K), kTileK, kTileTok);
    if (st != TRDQ_OK) return st;
    st = encode_tmap_2d(&p.tmap_out[s], src.out, 2, static_cast<uint64_t>(w->N), static_cast<uint64_t>(src.M),
                        static_cast<uint64_t>(src.ld) * 2, 32, kTokPerWarp, 64);
    if (st != TRDQ_OK) return st;
  }
  for (int s = 0; s < 2; ++s) {
    if (seg[s].M > 0) continue;  // an empty segment's maps are never used, only prefetched: the other segment's
    p.tmap_a[s] = p.tmap_a[1 - s];
    p.tmap_out[s] = p.tmap_out[1 - s];
  }
  p.tmap_b = w->groups[g].tmap_b[0];
  p.mult_t = w->groups[g].mult_t;
  p.base = w->groups[g].base;
  p.bias = static_cast<const __nv_bfloat16*>(bias_bf16);
  p.N = w->N;
  p.K = w->K;
  p.tiles_n = (w->N + kTileCh - 1) / kTileCh;
  p.n_pad = p.tiles_n * kTileCh;
  p.fast_shift = kMultBits - w4_fast_bits(w->K / kTileK);
  p.status = device_status_word();
  if (!p.status) return TRDQ_ERR_CUDA;
  const int64_t total = tiles_m * p.tiles_n;
  const int grid = static_cast<int>(total < sms ? total : sms);
  static PerDeviceFlag configured;
  if (!configured.get(dev)) {
    for (const auto kernel : {gemm_w4a8_kernel<false, false>, gemm_w4a8_kernel<false, true>, gemm_w4a8_kernel<true, false>, gemm_w4a8_kernel<true, true>})
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) return TRDQ_ERR_CUDA;
    configured.set(dev, true);
  }
  // The kernel with both forms of the sum has 73 KB of instructions (98 with GELU) in place of 40 (53), more than stays cached when kernels alternate, as
  // the layers of a block do: its launch and the ones around it take 4 - 8 us longer than in a loop by themselves.  So it runs from 200 k-blocks per SM
  // on, where it gains 12 us and more.  A block of 4-bit layers, microseconds, 64-bit sums throughout / wherever the reduction is short / from here on: 1000 tokens of
  // width 384 41.1 / 45.6 / 41.3, 4000 of 896 164.3 / 171.5 / 161.9, 2000 of 1152 with cross-attention 171 / 180 / 170, 16384 of 1152 738 / 728 / 730, of 768 414 / - / 406.
  const int64_t blocks = w->K / kTileK;
  const bool fast = w4_fast_bits(static_cast<int>(blocks)) >= kMinFastBits && total * blocks >= kFastBlocksPerSm * sms;
  void (*const kernel)(W4Params) = act ? (fast ? gemm_w4a8_kernel<true, true> : gemm_w4a8_kernel<true, false>)
                                       : (fast ? gemm_w4a8_kernel<false, true> : gemm_w4a8_kernel<false, false>);
  const cudaError_t e = launch_overlapped(kernel, dim3(grid), dim3(kThreads), kSmemBytes, stream, p);
  return e == cudaSuccess ? TRDQ_OK : TRDQ_ERR_CUDA;
}

}  // namespace trdq
