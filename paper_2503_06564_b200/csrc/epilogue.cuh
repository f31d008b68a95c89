// Dequantizing epilogue arithmetic shared by the 8-bit GEMM kernels (Eq. 10 on the codes, then the
// per-token and per-channel scales of Sec. 3.1 and the bias).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace trdq {

// One output: y = acc * sx * sw + bias in fp32.  fp32 is accurate to 2^-23 of the product; only when
// product and bias cancel below `thr` = 2^-10 |bias| can that exceed a bf16 rounding step of the result;
// then the scale product is carried as an exact two-term sum and the part of the accumulator that
// fp32 could not hold is added back (to v, the value without these two parts).
__device__ __forceinline__ float repair_cancellation(int32_t a, float sxm, float swn, float v) {
  const float af = static_cast<float>(a);
  const float s_hi = __fmul_rn(sxm, swn);
  const float s_lo = __fmaf_rn(sxm, swn, -s_hi);
  v = __fmaf_rn(af, s_lo, v);
  return __fmaf_rn(static_cast<float>(a - __float2int_rz(af)), s_hi, v);
}
__device__ __forceinline__ float dequant_one(int32_t a, float sxm, float swn, float biasn, float thr) {
  const float v = __fmaf_rn(static_cast<float>(a), __fmul_rn(sxm, swn), biasn);
  return fabsf(v) < thr ? repair_cancellation(a, sxm, swn, v) : v;
}

// GELU in its tanh form, the activation between the two MLP linears of a DiT block, two values at a time:
//   gelu(x) = 0.5 x (1 + tanh(u)) = x / (1 + exp(-2u)) = x exp(2u) / (1 + exp(2u)),   u = sqrt(2/pi) (x + 0.044715 x^3).
// With e = exp(-|2u|) in [0, 1] the denominator d = 1 + e stays in [1, 2] on both sides, so nothing overflows and the
// flush-to-zero form of 1 / x is in its defined range.  2^x keeps subnormal results: e is one from x = -10.0 down, and x e then
// still is a number that bf16 holds (to x = -10.6).
// (The form of 2^x that keeps subnormals takes three more instructions, so gelu_pack uses it only where it makes a difference.  One reciprocal
// shared by four quotients would move one bf16 result in 10^5, and repairing those costs more than is gained.)
template <bool FLUSH>
__device__ __forceinline__ float exp2_approx(float x) {
  float r;
  if constexpr (FLUSH) {
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  } else {
    asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  }
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <bool FLUSH>
__device__ __forceinline__ float2 gelu_tanh2(float2 x) {
  const float k = 1.5957691216057308f;  // 2 sqrt(2/pi)
  const float log2e = 1.4426950408889634f;
  const float2 t = __fmul2_rn(x, __ffma2_rn(__fmul2_rn(x, x), make_float2(0.044715f * k, 0.044715f * k), make_float2(k, k)));  // 2u, sign of x
  const float2 t2 = __fmul2_rn(t, make_float2(log2e, log2e));
  const float2 e = make_float2(exp2_approx<FLUSH>(-fabsf(t2.x)), exp2_approx<FLUSH>(-fabsf(t2.y)));
  const float2 m = __fmul2_rn(x, e);
  const float2 d = __fadd2_rn(e, make_float2(1.0f, 1.0f));
  return __fmul2_rn(make_float2(t.x >= 0.0f ? x.x : m.x, t.y >= 0.0f ? x.y : m.y), make_float2(rcp_ftz(d.x), rcp_ftz(d.y)));
}

__device__ __forceinline__ uint32_t pack_bf16(float2 v) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// GELU of 2 PAIRS values, packed to bf16.  One test for all of them: from -9.75 up 2^x is a normal number and both forms of it agree.
// For kernels that issue more than they wait, the CTA-pair GEMM: 1152 -> 4608 with GELU, without / with the test, 22.8 -> 22.1 us at M = 4096, 79.4 -> 76.7
// at 16384.  Where a CTA has one or two tiles the test only adds to the last epilogue (single-CTA GEMM, N x M: K = 1152, 1152 x 700 5.74 -> 5.94 us,
// K = 4608, 384 x 1400 9.84 -> 10.06), and the 4-bit kernel is no faster with it (264 -> 269).
template <int PAIRS>
__device__ __forceinline__ void gelu_pack(const float2 (&v)[PAIRS], uint32_t (&packed)[PAIRS]) {
  float lowest = v[0].x;
#pragma unroll
  for (int j = 0; j < PAIRS; ++j) asm("min.f32 %0, %0, %1, %2;" : "+f"(lowest) : "f"(v[j].x), "f"(v[j].y));
  if (lowest < -9.75f) {
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) packed[j] = pack_bf16(gelu_tanh2<false>(v[j]));
  } else {
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) packed[j] = pack_bf16(gelu_tanh2<true>(v[j]));
  }
}

// min(|a|, |b|, |c|) in one instruction
__device__ __forceinline__ float min3_abs(float a, float b, float c) {
  float r;
  asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Epilogue parameters of a tile in shared memory: per column the weight scale and the bias, per eight columns the
// largest cancellation threshold 2^-10 |bias| among them.
struct ColumnParams {
  const float* sw;
  const float* bias;
  const float* thr;
};
template <int BN>
struct ColumnParamLayout {  // [sw BN][bias BN][thr BN / 8], 16-byte aligned
  static constexpr int kFloats = 2 * BN + BN / 8;
  static constexpr int kBytes = kFloats * 4;
};

enum EpilogueAct { kActNone, kActGelu, kActGeluTested };  // kActGeluTested: through gelu_pack

// COLS (16 or 32) consecutive columns (the c-th such group of the tile) of one output row: y = acc * sx * sw[n] + bias[n] (then GELU, see ACT),
// packed to bf16 pairs.  Packed fp32x2 arithmetic, the same roundings as dequant_one; the cancellation against the bias is
// looked for once per row and eight columns (smallest |y| against the largest threshold of the eight).  Where it may have
// happened the eight are held against their own thresholds, and only those below are repaired: with a bias of the output's size a
// value in 10^3 is below the largest threshold, so in a warp of 32 rows every third or fourth group of eight columns, but hardly one below its own.
// Microseconds of the GEMM with each column tested by itself / one test per 32 columns that repairs all of them / this, for a bias
// of a hundredth of the output's size and one of twice its size: M = 4096, 1152 -> 4608 19.1 / 17.1 / 17.4 and 19.1 / 20.7 / 18.4, M = 16384,
// 1152 -> 3456 54.7 / 52.7 / 51.7 and 54.5 / 59.4 / 52.9.  One test per four columns costs more than it saves (17.3 and 19.8).
template <int COLS, EpilogueAct ACT>
__device__ __forceinline__ void dequant_row(const uint32_t (&r)[COLS], float sxm, const ColumnParams& cp, int c, uint32_t (&packed)[COLS / 2]) {
  static_assert(COLS == 16 || COLS == 32, "two or four tests");
  const float4* sw4 = reinterpret_cast<const float4*>(cp.sw + c * COLS);
  const float4* b4 = reinterpret_cast<const float4*>(cp.bias + c * COLS);
  const float2 sx2 = make_float2(sxm, sxm);
  float2 v[COLS / 2];
  float low[4];
#pragma unroll
  for (int j = 0; j < COLS / 4; ++j) {
    const float4 s = sw4[j], b = b4[j];
    const float2 a0 = make_float2(static_cast<float>(static_cast<int32_t>(r[4 * j])), static_cast<float>(static_cast<int32_t>(r[4 * j + 1])));
    const float2 a1 = make_float2(static_cast<float>(static_cast<int32_t>(r[4 * j + 2])), static_cast<float>(static_cast<int32_t>(r[4 * j + 3])));
    v[2 * j] = __ffma2_rn(a0, __fmul2_rn(sx2, make_float2(s.x, s.y)), make_float2(b.x, b.y));
    v[2 * j + 1] = __ffma2_rn(a1, __fmul2_rn(sx2, make_float2(s.z, s.w)), make_float2(b.z, b.w));
    low[j / 2] = min3_abs(j & 1 ? low[j / 2] : __uint_as_float(0x7F800000u), v[2 * j].x, v[2 * j].y);
    low[j / 2] = min3_abs(low[j / 2], v[2 * j + 1].x, v[2 * j + 1].y);
  }
  float4 thr;
  if constexpr (COLS == 32) {
    thr = *reinterpret_cast<const float4*>(cp.thr + c * 4);
  } else {
    const float2 two = *reinterpret_cast<const float2*>(cp.thr + c * 2);
    thr = make_float4(two.x, two.y, 0.0f, 0.0f);
  }
  // not "low < thr": also when a NaN bias made the threshold one
  const bool cancels[4] = {!(low[0] >= thr.x), !(low[1] >= thr.y), COLS == 32 && !(low[2] >= thr.z), COLS == 32 && !(low[3] >= thr.w)};
  if (cancels[0] || cancels[1] || cancels[2] || cancels[3]) {
#pragma unroll
    for (int g = 0; g < COLS / 8; ++g) {
      if (!cancels[g]) continue;
      const float4 b0 = b4[2 * g], b1 = b4[2 * g + 1];
      const float bn[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
      bool own = false;
#pragma unroll
      for (int e = 0; e < 8; ++e) own |= fabsf(e & 1 ? v[4 * g + e / 2].y : v[4 * g + e / 2].x) < fabsf(bn[e]) * 0.0009765625f;
      if (!own) continue;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int j = 8 * g + e;
        float& y = j & 1 ? v[j / 2].y : v[j / 2].x;
        if (fabsf(y) < fabsf(bn[e]) * 0.0009765625f) y = repair_cancellation(static_cast<int32_t>(r[j]), sxm, cp.sw[c * COLS + j], y);
      }
    }
  }
  if constexpr (ACT == kActGeluTested) {
    gelu_pack(v, packed);
  } else {
#pragma unroll
    for (int j = 0; j < COLS / 2; ++j) packed[j] = pack_bf16(ACT == kActGelu ? gelu_tanh2<false>(v[j]) : v[j]);
  }
}

// Staging of the epilogue parameters of BN columns (see ColumnParamLayout): the scale and bias of column n, then their place c in the
// tile's table.  store_column_param is called by whole warps with consecutive c: a warp holds whole groups of eight columns.
// Columns from N on (their outputs are clipped by the store) get an infinite bias and no threshold: with zeros their outputs would be 0
// and every row of a chunk that N ends in would look like a cancellation.
struct ColumnParam {  // scale and bias of one column
  float s, b;
};
__device__ __forceinline__ ColumnParam load_column_param(const float* sw, const __nv_bfloat16* bias, int n, int N) {
  ColumnParam c{0.0f, __uint_as_float(0x7F800000u)};
  if (n < N) {
    c.s = __ldg(sw + n);
    c.b = bias ? __bfloat162float(bias[n]) : 0.0f;
  }
  return c;
}
template <int BN>
__device__ __forceinline__ void store_column_param(float* dst, const ColumnParam& v, bool inside, int c) {
  // non-negative floats order like their bit patterns (a NaN bias gives a NaN threshold)
  unsigned int top = inside ? __float_as_uint(fabsf(v.b) * 0.0009765625f) : 0u;
  dst[c] = v.s;
  dst[BN + c] = v.b;
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, d));
  if ((c & 7) == 0) dst[2 * BN + c / 8] = __uint_as_float(top);
}

// The parameters of a tile of 128 rows and BN columns: [columns (ColumnParamLayout)][weight column sums BN][row scales 128][zero points 128].
constexpr int kParamRows = 128;
template <int BN>
struct TileParams {
  static constexpr int kBytes = ColumnParamLayout<BN>::kBytes + BN * 4 + 2 * kParamRows * 4;
  ColumnParams columns;
  int32_t* colsum;
  float* sx;
  int32_t* zp;
  __device__ __forceinline__ explicit TileParams(uint8_t* base) {
    float* const f = reinterpret_cast<float*>(base);
    columns = ColumnParams{f, f + BN, f + 2 * BN};
    colsum = reinterpret_cast<int32_t*>(f + ColumnParamLayout<BN>::kFloats);
    sx = reinterpret_cast<float*>(colsum + BN);
    zp = reinterpret_cast<int32_t*>(sx + kParamRows);
  }
};
// Called by two whole warps, st = 0 .. 63; `wait_free` returns once the set may be overwritten, the loads are in flight meanwhile.
template <int BN, bool ASYM, typename Wait>
__device__ __forceinline__ void stage_tile_params(uint8_t* set, const float* sw, const __nv_bfloat16* bias, const int32_t* colsum, int n0, int N,
                                                  const float* sx, const int32_t* zp, int m0, int M, int st, Wait&& wait_free) {
  ColumnParam col[BN / 64];
  int32_t csum[BN / 64], zr[kParamRows / 64];
  float sxr[kParamRows / 64];
#pragma unroll
  for (int i = 0; i < BN / 64; ++i) {
    const int n = n0 + 64 * i + st;
    col[i] = load_column_param(sw, bias, n, N);
    if (ASYM) csum[i] = n < N ? __ldg(colsum + n) : 0;
  }
#pragma unroll
  for (int i = 0; i < kParamRows / 64; ++i) {
    const int row = m0 + 64 * i + st;
    sxr[i] = row < M ? __ldg(sx + row) : 0.0f;
    if (ASYM) zr[i] = row < M ? __ldg(zp + row) : 0;
  }
  wait_free();
  const TileParams<BN> t(set);
#pragma unroll
  for (int i = 0; i < BN / 64; ++i) {
    store_column_param<BN>(reinterpret_cast<float*>(set), col[i], n0 + 64 * i + st < N, 64 * i + st);
    if (ASYM) t.colsum[64 * i + st] = csum[i];
  }
#pragma unroll
  for (int i = 0; i < kParamRows / 64; ++i) {
    t.sx[64 * i + st] = sxr[i];
    if (ASYM) t.zp[64 * i + st] = zr[i];
  }
}

// The columns of a tile that starts at column n0, by the threads tid = 0 .. nthreads - 1, nthreads a multiple of 32.
template <int BN>
__device__ __forceinline__ ColumnParams stage_column_params(float* dst, const float* sw, const __nv_bfloat16* bias, int n0, int N, int tid,
                                                            int nthreads) {
  for (int c = tid; c < BN; c += nthreads) store_column_param<BN>(dst, load_column_param(sw, bias, n0 + c, N), n0 + c < N, c);
  return ColumnParams{dst, dst + BN, dst + 2 * BN};
}

}  // namespace trdq
