// Pieces shared by the kernels that give one thread a whole 128-block of one row (128 fp32 values in registers) and split
// the CTA into teams of warps that hold whole rows.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lane_group.cuh"
#include "ptx.cuh"

namespace trdq {

constexpr int kTeamMaxWarps = 12;    // 12 x 32 threads x <= 168 registers fill the register file
constexpr int kVecPadFloats = 4;     // a per-channel table of block b starts at float b * (128 + 4): see stage_vector

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

// max(|a|, |b|, |c|) in one instruction
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float r;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ void team_barrier(int team, int team_threads) {
  if (team_threads == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(team_threads) : "memory");
}

// A per-channel table of K floats, block b at float b * 132: lanes of a quarter warp that hold different blocks then read
// different bank groups with their 16-byte loads (same block: same address, a broadcast).
__device__ __forceinline__ void stage_vector(float* dst, const float* src, int K) {
  // not unrolled: most threads take one or two turns, and the unrolled loop's preamble costs a launch 0.1 us (K = 1152: 3.26 -> 3.38 at
  // M = 1480, 7.59 -> 7.83 at 8192)
#pragma unroll 1
  for (int i = threadIdx.x; i < K / 4; i += blockDim.x) {
    const int b = i >> 5;
    reinterpret_cast<float4*>(dst + b * (TRDQ_BLOCK + kVecPadFloats))[i & 31] = __ldg(reinterpret_cast<const float4*>(src) + i);
  }
}

// The thread's block (row r, block b) of a TMA-staged bf16 tile: column boxes of 64, each R rows of 128 bytes, 128-byte
// swizzle, times the fused vector sv4 of the block.  v[32h + 4j + i] = elements (2i, 2i+1) of 16-byte chunk j of half h.
__device__ __forceinline__ void load_scaled_block(uint32_t tile_base, uint32_t box_bytes, int b, int r, const float4* sv4, float2 (&v)[64]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t in_row = tile_base + (2 * b + h) * box_bytes + r * 128;
    const uint32_t swz = (in_row >> 7) & 7u;  // 128-byte swizzle: chunk index xor address bits 7..9
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4 raw = lds128(in_row + ((j ^ swz) << 4));
      const float4 s0 = sv4[h * 16 + j * 2], s1 = sv4[h * 16 + j * 2 + 1];
      const uint32_t wd[4] = {raw.x, raw.y, raw.z, raw.w};
      const float2 sc[4] = {make_float2(s0.x, s0.y), make_float2(s0.z, s0.w), make_float2(s1.x, s1.y), make_float2(s1.z, s1.w)};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // bf16 -> fp32 is exact: the 16 bits become the high half of the fp32 pattern
        const float2 xv = make_float2(__uint_as_float(wd[i] << 16), __uint_as_float(wd[i] & 0xFFFF0000u));
        v[h * 32 + j * 4 + i] = __fmul2_rn(xv, sc[i]);
      }
    }
  }
}

// 128-point unnormalised Walsh-Hadamard transform of a thread's block: stages h = 1 .. 64 in this order with separately
// rounded additions (h = 1 inside a pair, h = 2 .. 64: pair index bits 0 .. 5).
__device__ __forceinline__ void wht128_thread(float2 (&v)[64]) {
  const float2 neg1 = make_float2(-1.0f, -1.0f);
#pragma unroll
  for (int q = 0; q < 64; ++q) v[q] = make_float2(__fadd_rn(v[q].x, v[q].y), __fsub_rn(v[q].x, v[q].y));
#pragma unroll
  for (int hb = 1; hb < 64; hb <<= 1) {
#pragma unroll
    for (int q = 0; q < 64; ++q) {
      if ((q & hb) == 0) {
        const float2 a = v[q], c = v[q + hb];
        v[q] = __fadd2_rn(a, c);
        v[q + hb] = __ffma2_rn(c, neg1, a);  // a - c, one rounding
      }
    }
  }
}

__device__ __forceinline__ float absmax_thread(const float2 (&v)[64]) {
  float m = 0.0f;
#pragma unroll
  for (int q = 0; q < 64; ++q) m = max3_abs(m, v[q].x, v[q].y);
  return m;
}

// Symmetric int8 codes of the thread's block to its 128 swizzled bytes of the code tile: q = rne(fl(v * inv)).
// The product must be rounded to fp32 before the magic addition rounds it to an integer.  A packed multiply feeding a
// packed add is contracted into one fused operation by the assembler, so the product is written as fma(v, inv, zero) with
// `zero` a kernel argument equal to 0.0f.
__device__ __forceinline__ void quantize_store_block(const float2 (&v)[64], float inv, float zero, uint32_t out_row) {
  const float2 inv2 = make_float2(inv, inv), magic2 = make_float2(kRoundMagic, kRoundMagic), zero2 = make_float2(zero, zero);
  const uint32_t oswz = (out_row >> 7) & 7u;
#pragma unroll
  for (int c = 0; c < 8; ++c) {  // 16 codes = 8 pairs per 16-byte chunk
    float2 q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = __fadd2_rn(__ffma2_rn(v[c * 8 + i], inv2, zero2), magic2);
    st_shared_v4(out_row + ((c ^ oswz) << 4), pack4(q[0], q[1]), pack4(q[2], q[3]), pack4(q[4], q[5]), pack4(q[6], q[7]));
  }
}

}  // namespace trdq
