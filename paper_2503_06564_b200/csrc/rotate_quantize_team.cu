// Fused online transform + per-token quantizer (Sec. 3.2 Eq. 10 G_t; Sec. 3.1 Eq. 1-2): TMA-staged input, ONE THREAD
// PER 128-BLOCK, and the CTA split into small TEAMS that each run their own pipeline.
//
// A thread holds a whole block (128 fp32 values in registers), so all seven butterfly stages are register-to-register
// packed fp32x2 operations.  That costs ~160 registers per thread, i.e. at most twelve warps per SM, so latency cannot be
// hidden by occupancy.  It is hidden by letting the warps run out of phase instead: a team is the smallest group of warps
// that holds whole rows (K = 1152: one warp = 3 rows of 9 blocks, 27 of 32 lanes; K = 4608: five warps = 4 rows of 36
// blocks, 144 of 160 lanes), and every team has its own two-stage TMA ring, its own row-maximum exchange, its own code
// staging tile and its own named barrier.  Nothing synchronises two teams, so while one waits for data or for its row
// maximum the others transform; there is no producer warp (lane 0 of a team refills the stage its team has just read).
//
// The arithmetic (one fp32 multiply by the fused vector, stages h = 1 .. 64 in this order with separately rounded
// additions, rne via the 1.5 * 2^23 addition) is the same as in the other kernels of rotate_quantize.cu and
// bit-identical to a scalar evaluation.  Every wait is bounded.
#include <cuda_bf16.h>

#include "internal.h"
#include "team.cuh"

namespace trdq {
namespace {

struct alignas(64) TeamParams {
  // Both maps view a row as K/64 (K/128) column boxes: dims (column in box, row, box), so that ONE copy moves a tile of R
  // whole rows and lays it out box after box, each box R rows of 128 bytes, 128-byte swizzle.
  CUtensorMap tmap_x;      // bf16: (64, M, K/64), box 64 x R x K/64
  CUtensorMap tmap_codes;  // int8: (128, M, K/128), box 128 x R x K/128
  const float* vec;        // fused vector of the group, K floats
  float* scales;           // [M]
  int32_t* zero_points;    // [M], asymmetric form only
  int32_t M, K;
  int32_t R;               // rows per team tile
  int32_t team_warps;      // warps per team (R * K/128 <= 32 * team_warps)
  int32_t teams;           // teams per CTA
  float zero;              // 0.0f, see quantize_store_block
  uint32_t* status;
};

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Unsigned codes of the thread's block (Eq. 1-3): code = min(rne(fl(v * inv)) + z, 255); the lower clamp of Eq. 1 can never bind
// (rounding is monotone and z cancels the minimum's own code).  fl(v * inv) + 1.5 * 2^23 leaves the rounded product in the low
// mantissa bits; adding z and the clamp are exact there as long as |v * inv| < 2^22, which `small` says for the whole row.
// Other rows (a range so narrow or so wide that 255 / range or the products leave the integers, NaN) take the integer form of the
// lane-group kernel word for word: which of the two kernels a call runs depends on M and may not show in its codes.
__device__ __forceinline__ void quantize_store_block_asym(const float2 (&v)[64], float inv, int z, bool small, float zero, uint32_t out_row) {
  const uint32_t oswz = (out_row >> 7) & 7u;
  if (!small) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      uint32_t wd[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int q0 = min(__float2int_rn(__fmul_rn(v[c * 8 + i].x, inv)) + z, 255);
        const int q1 = min(__float2int_rn(__fmul_rn(v[c * 8 + i].y, inv)) + z, 255);
        wd[i / 2] |= (static_cast<uint32_t>(q0) | (static_cast<uint32_t>(q1) << 8)) << (16 * (i & 1));
      }
      st_shared_v4(out_row + ((c ^ oswz) << 4), wd[0], wd[1], wd[2], wd[3]);
    }
    return;
  }
  const float2 inv2 = make_float2(inv, inv), magic2 = make_float2(kRoundMagic, kRoundMagic), zero2 = make_float2(zero, zero);
  const float zf = static_cast<float>(z);
  const float2 z2 = make_float2(zf, zf);
  constexpr float top = kRoundMagic + 255.0f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float2 q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 u = __fadd2_rn(__fadd2_rn(__ffma2_rn(v[c * 8 + i], inv2, zero2), magic2), z2);
      q[i] = make_float2(fminf(u.x, top), fminf(u.y, top));
    }
    st_shared_v4(out_row + ((c ^ oswz) << 4), pack4(q[0], q[1]), pack4(q[2], q[3]), pack4(q[4], q[5]), pack4(q[6], q[7]));
  }
}

// ASYM: the literal asymmetric quantizer of Eq. 1-3 (row minimum and maximum, unsigned codes, a zero point per row).
template <bool ASYM>
__global__ void __launch_bounds__(kTeamMaxWarps * 32, 1) rotate_quantize_team_kernel(const __grid_constant__ TeamParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 127u) & ~127u;  // TMA destinations need 128 bytes; the swizzle is a function of the address
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  const int nb = p.K / TRDQ_BLOCK;
  const int R = p.R;
  const uint32_t box_bytes = R * 128;             // one column box: R rows of 128 bytes
  const uint32_t in_bytes = 2 * nb * box_bytes;   // R x K bf16
  const uint32_t out_bytes = nb * box_bytes;      // R x K int8
  const uint32_t team_bytes = 2 * in_bytes + out_bytes;
  float* svec = reinterpret_cast<float*>(smem + p.teams * team_bytes);
  unsigned int* row_max_all = reinterpret_cast<unsigned int*>(svec + nb * (TRDQ_BLOCK + kVecPadFloats));  // [teams][3][R]
  uint64_t* bars = reinterpret_cast<uint64_t*>(row_max_all + (ASYM ? 2 * p.teams * 3 * R : (p.teams * 3 * R + 1) & ~1));  // [teams][2]

  const int tid = threadIdx.x;
  const int team_threads = p.team_warps * 32;
  const int team = tid / team_threads;
  const int tt = tid - team * team_threads;
  const uint32_t team_base = smem_base + team * team_bytes;
  const uint32_t out_base = team_base + 2 * in_bytes;
  unsigned int* row_max = row_max_all + team * 3 * R;
  unsigned int* row_min = row_max + p.teams * 3 * R;  // ASYM: keys of the minima behind those of the maxima
  const uint32_t bar_full = smem_u32(bars + 2 * team);  // [2]

  if (tt == 0) {
    mbar_init(bar_full, 1);
    mbar_init(bar_full + 8, 1);
    fence_mbar_init();
  }
  stage_vector(svec, p.vec, p.K);
  for (int i = tid; i < p.teams * 3 * R; i += blockDim.x) {
    row_max_all[i] = 0u;
    if (ASYM) row_max_all[p.teams * 3 * R + i] = 0xFFFFFFFFu;
  }
  if (tid == 0) {
    prefetch_tensormap(&p.tmap_x);
    prefetch_tensormap(&p.tmap_codes);
  }
  __syncthreads();
  griddep_launch_dependents();
  griddep_wait();  // X may be written, and the code buffer still read, by the kernel before (the group vector is constant)

  // Tiles of R rows are dealt to the teams of the whole grid, SM after SM, so that the teams with one tile more than
  // the others are spread over all SMs.
  const int num_tiles = (p.M + R - 1) / R;
  const int stride = gridDim.x * p.teams;
  const int first = team * gridDim.x + blockIdx.x;
  // Only the FIRST tile of every team is requested here; the second one follows when the first has landed (below).  All
  // teams of all CTAs start together, so asking for both at once doubles the burst every first tile has to wait behind.
  if (tt == 0 && first < num_tiles) {
    mbar_arrive_expect_tx(bar_full, in_bytes);
    tma_load_3d(team_base, &p.tmap_x, 0, first * R, 0, bar_full);  // all 2 * nb column boxes in one copy
  }

  // consecutive threads = consecutive rows of one block column
  const bool active = tt < R * nb;
  const int b = active ? tt / R : 0;
  const int r = active ? tt - b * R : 0;
  const float4* sv4 = reinterpret_cast<const float4*>(svec + b * (TRDQ_BLOCK + kVecPadFloats));

  BoundedWaiter w(p.status, kStatusTimeoutEpilogue);
  int it = 0;
  for (int tile = first; tile < num_tiles; tile += stride, ++it) {
    const int s = it & 1;
    const uint32_t phase = (it >> 1) & 1;
    const int buf = it % 3;
    if (tt < R) {
      row_max[((it + 1) % 3) * R + tt] = 0u;
      if (ASYM) row_min[((it + 1) % 3) * R + tt] = 0xFFFFFFFFu;
    }

    w.wait(bar_full + 8 * s, phase);
    if (it == 0 && tt == 0 && tile + stride < num_tiles) {  // the team's second tile, into the other stage
      mbar_arrive_expect_tx(bar_full + 8, in_bytes);
      tma_load_3d(team_base + in_bytes, &p.tmap_x, 0, (tile + stride) * R, 0, bar_full + 8);
    }
    float2 v[64];
    load_scaled_block(team_base + s * in_bytes, box_bytes, b, r, sv4, v);
    wht128_thread(v);
    if (ASYM) {
      float hi = v[0].x, lo = v[0].x;
#pragma unroll
      for (int q = 0; q < 64; ++q) {
        hi = max3(hi, v[q].x, v[q].y);
        lo = min3(lo, v[q].x, v[q].y);
      }
      if (active) {
        atomicMax(&row_max[buf * R + r], float_order_key(hi));
        atomicMin(&row_min[buf * R + r], float_order_key(lo));
      }
    } else {
      const float m = absmax_thread(v);
      if (active) atomicMax(&row_max[buf * R + r], __float_as_uint(m));
    }
    if (tt == 0) bulk_wait_group_read<0>();  // the previous tile's store has finished reading the staging tile
    team_barrier(team, team_threads);        // row maxima complete; every thread of the team has read stage s

    if (tt == 0) {
      const int next = tile + 2 * stride;
      if (next < num_tiles) {
        mbar_arrive_expect_tx(bar_full + 8 * s, in_bytes);
        tma_load_3d(team_base + s * in_bytes, &p.tmap_x, 0, next * R, 0, bar_full + 8 * s);
      }
    }

    const int64_t row = static_cast<int64_t>(tile) * R + r;
    const uint32_t out_row = out_base + b * box_bytes + r * 128;
    if (ASYM) {
      const float vmax = float_from_order_key(row_max[buf * R + r]);
      const float vmin = float_from_order_key(row_min[buf * R + r]);
      const float range = __fsub_rn(vmax, vmin);
      const float inv = range > 0.0f ? __fdiv_rn(255.0f, range) : 0.0f;
      const int z = -__float2int_rn(__fmul_rn(vmin, inv));
      // false also where infinities or NaN took part (a NaN input makes the block's sum v[0].x one)
      const bool small = fmaxf(fabsf(vmax), fabsf(vmin)) * inv < 4194303.0f && v[0].x == v[0].x;
      if (active) {
        quantize_store_block_asym(v, inv, z, small, p.zero, out_row);
        if (b == 0 && row < p.M) {
          p.scales[row] = __fdiv_rn(range, 255.0f);
          p.zero_points[row] = z;
        }
      }
    } else {
      const float amax = __uint_as_float(row_max[buf * R + r]);
      const float inv = amax > 0.0f ? __fdiv_rn(127.0f, amax) : 0.0f;
      if (active) {
        quantize_store_block(v, inv, p.zero, out_row);
        if (b == 0 && row < p.M) p.scales[row] = __fdiv_rn(amax, 127.0f);
      }
    }
    fence_proxy_async_smem();
    team_barrier(team, team_threads);
    if (tt == 0) {
      tma_store_3d(&p.tmap_codes, 0, tile * R, 0, out_base);  // all nb column boxes; rows >= M are clipped
      bulk_commit_group();
    }
  }
  if (tt == 0) bulk_wait_group_read<0>();  // the staging tile has been read; the stores complete before the grid does
  w.settle();
}

// One row-exchange table (three buffers of the row maxima), in the asymmetric form two (the minima as well): charging both to the
// symmetric form would cost it a team at K = 128, eleven against ten.
size_t team_smem_bytes(int K, int R, int teams, bool asym) {
  const int nb = K / TRDQ_BLOCK;
  return 128 + static_cast<size_t>(teams) * 5 * R * K + static_cast<size_t>(nb) * (TRDQ_BLOCK + kVecPadFloats) * 4 +
         (static_cast<size_t>(teams) * (asym ? 6 : 3) * R + 2) * 4 + static_cast<size_t>(teams) * 16 + 16;
}

// The team of `tw` warps for rows of K channels: as many whole rows as its lanes hold, as many teams as registers
// (twelve warps) and shared memory (two input stages and a code tile per team) allow.  At least two teams, so that one
// can transform while another waits.
bool team_shape_for(int K, int tw, bool asym, TeamShape* out) {
  const int nb = K / TRDQ_BLOCK;
  int rows = tw * 32 / nb;
  if (rows < 1) return false;
  if (rows > 32) rows = 32;
  int teams = kTeamMaxWarps / tw;
  while (teams > 0 && team_smem_bytes(K, rows, teams, asym) > 227u * 1024u) --teams;
  if (teams < 2) return false;
  *out = TeamShape{rows, tw, teams, team_smem_bytes(K, rows, teams, asym),
                   static_cast<double>(rows) * nb / (tw * 32) * (static_cast<double>(teams * tw) / kTeamMaxWarps)};
  return true;
}

int device_sm_count(int* dev_out) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (dev_out) *dev_out = dev;
  return sms;
}

}  // namespace

// Team size by lane use (K = 1152: one warp, 3 rows, 27 of 32 lanes, twelve teams; K = 4608: four warps, 3 rows, 108 of
// 128 lanes, three teams).  With fewer than about one tile per team the next larger team is taken when the best one
// is a single warp: fewer, fatter tiles finish sooner when nothing is left to overlap (K = 1152, M = 4096: 6.2 against
// 6.7 us, measured).
bool rotate_quantize_team_shape(int M, int K, int sms, bool asym, TeamShape* out) {
  TeamShape best = {0, 0, 0, 0, 0.0};
  for (int tw = 1; tw <= kTeamMaxWarps / 2; ++tw) {
    TeamShape s;
    if (team_shape_for(K, tw, asym, &s) && s.use > best.use + 1e-9) best = s;
  }
  if (best.teams == 0) return false;
  const int64_t tiles = (static_cast<int64_t>(M) + best.R - 1) / best.R;
  TeamShape wider;
  if (best.team_warps == 1 && 4 * tiles < 5ll * best.teams * sms && team_shape_for(K, 2, asym, &wider)) best = wider;
  *out = best;
  return true;
}

// The team kernel serves rows for which at least two teams fit in shared memory, once there is at least a tile per SM; below
// that the lane-group kernel, whose CTAs are smaller and start sooner, finishes first (M = 256, K = 1024: 2.3 against 3.3 us).
static bool a_tile_per_sm(int32_t M, int32_t K, bool asym) {
  const int sms = device_sm_count(nullptr);
  TeamShape s;
  if (sms <= 0 || !rotate_quantize_team_shape(M, K, sms, asym, &s)) return false;
  return (static_cast<int64_t>(M) + s.R - 1) / s.R >= sms;
}
bool rotate_quantize_prefers_team(int32_t M, int32_t K) { return a_tile_per_sm(M, K, false); }

// Asymmetric codes: the second reduction over the block (minimum beside maximum) and its exchange make a team's tile longer, so
// the lane-group kernel keeps the smaller problems; and rows of more than 48 blocks, one or two to a team, need more of them still.
// Microseconds, lane groups / teams: K = 1152 at M = 2048 3.3 / 4.2, 8192 10.7 / 11.3, 16384 20.1 / 18.6, 32768 39.4 / 31.9;
// K = 2304 at 4096 11.9 / 11.5; K = 4608 at 2048 11.9 / 11.4, 4096 20.1 / 19.1, 8192 39.3 / 33.1; K = 6912 at 1639 13.5 / 14.2,
// 2304 17.5 / 18.2, 2891 21.5 / 20.3; K = 9216 at 1480 14.8 / 15.7, 2800 27.8 / 26.7;
// K = 9728 0.98 of the lane groups' speed from 2000 to 5000 rows and level at 12288, so from there on they keep every size.
bool rotate_quantize_asym_prefers_team(int32_t M, int32_t K) {
  if (K > 9216) return false;
  const int64_t least = K > 8192 ? 28ll << 20 : K > 6144 ? 16ll << 20 : K >= 2048 ? 9ll << 20 : 18ll << 20;
  return static_cast<int64_t>(M) * K >= least && a_tile_per_sm(M, K, true);
}

trdq_status launch_rotate_quantize_team(const void* x_bf16, int64_t ldx, int32_t M, int32_t K, const float* vec, void* codes,
                                        float* scales, int32_t* zero_points, cudaStream_t stream) {
  int dev = 0;
  const int sms = device_sm_count(&dev);
  if (sms <= 0) return TRDQ_ERR_CUDA;
  TeamShape shape;
  if (!rotate_quantize_team_shape(M, K, sms, zero_points != nullptr, &shape)) return TRDQ_ERR_SHAPE;
  const int nb = K / TRDQ_BLOCK;
  TeamParams p;
  trdq_status st = encode_tmap_boxes(&p.tmap_x, x_bf16, 2, 64, static_cast<uint64_t>(M), static_cast<uint64_t>(ldx) * 2,
                                     static_cast<uint32_t>(2 * nb), static_cast<uint32_t>(shape.R));
  if (st != TRDQ_OK) return st;
  st = encode_tmap_boxes(&p.tmap_codes, codes, 1, 128, static_cast<uint64_t>(M), static_cast<uint64_t>(K), static_cast<uint32_t>(nb),
                         static_cast<uint32_t>(shape.R));
  if (st != TRDQ_OK) return st;
  p.vec = vec;
  p.scales = scales;
  p.zero_points = zero_points;
  p.M = M;
  p.K = K;
  p.R = shape.R;
  p.team_warps = shape.team_warps;
  p.teams = shape.teams;
  p.zero = 0.0f;
  p.status = device_status_word();
  if (!p.status) return TRDQ_ERR_CUDA;
  static PerDeviceFlag configured;
  if (!configured.get(dev)) {
    if (cudaFuncSetAttribute(rotate_quantize_team_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
        cudaFuncSetAttribute(rotate_quantize_team_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
      return TRDQ_ERR_CUDA;
    configured.set(dev, true);
  }
  const int num_tiles = (M + shape.R - 1) / shape.R;
  const int grid = num_tiles < sms ? num_tiles : sms;  // few tiles: spread them over the SMs, fewer busy teams on each
  const cudaError_t e = launch_overlapped(zero_points ? rotate_quantize_team_kernel<true> : rotate_quantize_team_kernel<false>, dim3(grid), dim3(shape.teams * shape.team_warps * 32), shape.smem,
                                          stream, p);
  return e == cudaSuccess ? TRDQ_OK : TRDQ_ERR_CUDA;
}

}  // namespace trdq
