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
// What bounds it: the drain.  A 32 x 32 -> 64-bit multiply-add issues at a quarter of the fp32 rate: the drain loop by itself takes 603 clocks per k-block of
// 128 x 128 accumulators, 185 of them the loads from tensor memory, against 256 of tensor pipe.  In the kernel a k-block takes about 1100, and a tile 4000
// more for conversion and output.  M = 16384, microseconds with the weights as the N operand (multipliers read from a shared-memory table per
// column, one k-block per hand-over) -> now: 1152 -> 4608 323 -> 215 (with GELU 253), 4608 -> 1152 247 -> 166, 1152 -> 1152 84 -> 56, 1152 -> 3456 244 -> 163.
// Measured and not better: a CTA pair sharing the codes (1152 -> 4608 221 -> 211, but 1152 -> 1152 59 -> 64: the 256-channel tile pads N = 1152 by 11 %);
// sixteen drain warps of 32 tokens (218, 58); sums in fp64 (260 -> 358); weights unpacked into tensor memory with the codes of a token tile resident and one k-block
// per hand-over (221 -> 238, 4608 -> 1152 170 -> 180: four unpack warps and one instruction cache for everything); nibbles unpacked to q4 instead of
// 16 q4 (four more instructions per eight weights: 4608 -> 1152 170 -> 190).  The sum as two 32-bit numbers, its value modulo 2^32 and an fp32 sum
// in one binade (453 clocks), is exact to nine k-blocks and faster in a loop by itself (1152 -> 3456 163 -> 153), but only if its float is rounded twice; converted with one
// rounding it gives 159 - 168, and a block of four layers takes 743 - 771 in place of 731 (73 KB of instructions against 40).
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

constexpr int kMultBits = 30;

struct alignas(64) W4Params {
  CUtensorMap tmap_a[2];    // codes of each segment, box 128 B x 128 rows, 128-byte swizzle
  CUtensorMap tmap_b;       // packed weights, box 64 B x 64 rows
  CUtensorMap tmap_out[2];  // bf16 output, box 32 channels x 64 tokens, 64-byte swizzle
  const float* sx[2];
  int32_t M[2];
  int32_t tiles_m[2];
  const int32_t* mult_t;  // [K/128][n_pad]
  const float* base;      // [n_pad]
  const __nv_bfloat16* bias;
  int32_t N, K, tiles_n, n_pad;
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
// ACT: GELU (tanh form) on the dequantized value before the bf16 rounding.
template <bool ACT>
__device__ __forceinline__ void drain_tile(const W4Params& p, DrainState& s, int n, float base, float bias, int num_kb, const int32_t* next,
                                           const float (&sx_reg)[kTokPerWarp / 32]) {
  long long sum[kTokPerWarp];
#pragma unroll
  for (int j = 0; j < kTokPerWarp; ++j) sum[j] = 0;
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
    int32_t mult = s.m_next;
    asm volatile("" : "+r"(mult));  // stays a 32-bit factor: widened ahead of the loop it would cost a 64 x 64 product
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
      for (int j = 0; j < 16; ++j)
        sum[ch * 16 + j] += static_cast<long long>(static_cast<int32_t>(r[ch & 1][j])) * static_cast<long long>(mult);
    }
  }

  if (next) s.m_next = __ldg(next);
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
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __ll2float_rn(sum[j0 + e]);
    const float4 sa = *reinterpret_cast<const float4*>(s.sx + j0), sb = *reinterpret_cast<const float4*>(s.sx + j0 + 4);
    const float sx8[8] = {sa.x, sa.y, sa.z, sa.w, sb.x, sb.y, sb.z, sb.w};
    bool cancels = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      y[e] = __fmaf_rn(v[e], __fmul_rn(sx8[e], base), bias);
      cancels |= fabsf(y[e]) < thr;
    }
    if (cancels) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        // the part of the sum that fp32 dropped
        if (fabsf(y[e]) < thr) y[e] = __fmaf_rn(__ll2float_rn(sum[j0 + e] - __float2ll_rz(v[e])), __fmul_rn(sx8[e], base), y[e]);
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

// ACT: GELU (tanh form) on the dequantized value before the bf16 rounding.
template <bool ACT>
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
      drain_tile<ACT>(p, s, n, base, bias, num_kb, next, sx_reg);
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
  for (int g = 0; g < groups; ++g) {
    const float s = scales[static_cast<int64_t>(n) * groups + g];
    mult_t[static_cast<int64_t>(g) * n_pad + n] = __float2int_rn(ldexpf(s, kMultBits - e_max));  // < 2^30, exact if the exponents span < 7 bits
  }
  // the tensor core sees 16 * q4 (the nibble sits in the high half of the byte): fold the 1/16 here
  base[n] = ldexpf(1.0f, e_max - kMultBits - 4);
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
  p.status = device_status_word();
  if (!p.status) return TRDQ_ERR_CUDA;
  const int64_t total = tiles_m * p.tiles_n;
  const int grid = static_cast<int>(total < sms ? total : sms);
  static PerDeviceFlag configured;
  if (!configured.get(dev)) {
    for (const auto kernel : {gemm_w4a8_kernel<false>, gemm_w4a8_kernel<true>})
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) return TRDQ_ERR_CUDA;
    configured.set(dev, true);
  }
  const cudaError_t e = act ? launch_overlapped(gemm_w4a8_kernel<true>, dim3(grid), dim3(kThreads), kSmemBytes, stream, p)
                            : launch_overlapped(gemm_w4a8_kernel<false>, dim3(grid), dim3(kThreads), kSmemBytes, stream, p);
  return e == cudaSuccess ? TRDQ_OK : TRDQ_ERR_CUDA;
}

}  // namespace trdq
