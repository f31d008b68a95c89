// Full balancing transform (Eq. 9 / Eq. 10) + per-token quantizer, ONE THREAD PER 128-BLOCK, the CTA split into teams of
// warps that hold whole rows (see rotate_quantize_team.cu for the idea, team.cuh for the shared steps):
//     v1 = blockWHT(x o vec1),  v2[j] = fl32(v1[perm[j]] * vec2[j]),  v3 = blockWHT(v2),  codes of v3.
// Both butterflies are register-to-register.  Between them the rotated row is parked in shared memory as fp32, already
// times the second rotation's factor (vec2 is looked up at the SOURCE channel, where a whole block is written with 16-byte
// stores, instead of at each gathered value: the product is the same), and every thread gathers its 128 permuted channels;
// the table of byte offsets is 16 bits per channel, eight per load.
//
// What bounds it: the shared-memory pipe (per block and row some 30 wavefronts, for the most part the gather of 128 scalars at arbitrary
// banks) and the chain load - transform - barrier - gather - transform - maximum of a team, hidden only by other teams.  So it
// is rows in flight that count, and one buffer per team has to do for everything: the input tile lies in its first half until it is
// in registers, then the rotated rows take all of it, and the codes its last quarter, while the next input already arrives in the
// first half.  A separate input tile (requested most of a tile's time ahead) left room for 0.55 - 0.75 of the lanes of twelve warps; now
// it is 0.84 - 1.0.  Microseconds before -> now, M = 16384: K = 1152 27.9 -> 22.4, 1536 42.0 -> 26.4, 2304 58.2 -> 49.0, 3072 72.7 -> 53.6,
// 4608 115 -> 102; M = 4096: K = 1152 8.8 -> 7.8, 4608 33.4 -> 30.0, 7680 68.8 -> 54.5.  0.86 of the time over 401 points; five are slower by more than
// 1.5 %, where the larger tiles used before filled the last round better (K = 640 at M = 5000: 7.2 -> 7.8, K = 512 at 16384: 12.3 -> 12.7).
// The row buffer is swizzled (16-byte chunk index xor block) and rows are 48 bytes apart modulo 128, so that the writes of a
// quarter warp and the rows of one channel fall into different banks.
#include <cuda_bf16.h>

#include "internal.h"
#include "team.cuh"

namespace trdq {
namespace {

constexpr int kRowPadBytes = 48;

struct alignas(64) Team2Params {
  CUtensorMap tmap_x;      // bf16: (64, M, K/64), box 64 x R x K/64
  CUtensorMap tmap_codes;  // int8: (128, M, K/128), box 128 x R x K/128
  const float* vec1;       // fused vector of the group, K floats
  const int32_t* perm;     // (v P)[j] = v[perm[j]]
  const float* vec2;       // factors of the second rotation, by destination channel
  float* scales;           // [M]
  int32_t M, K;
  int32_t R, team_warps, teams;
  float zero;              // 0.0f, see quantize_store_block
  uint32_t* status;
};

// Byte offset of channel c inside a row of the row buffer.
__device__ __forceinline__ uint32_t row_offset(int c) {
  const int b = c >> 7;
  return static_cast<uint32_t>(b) * 512 + (((static_cast<uint32_t>(c) >> 2 & 31) ^ (b & 7)) << 4) + (c & 3) * 4;
}
__host__ __device__ constexpr uint32_t row_buffer_bytes(int K, int R) { return (static_cast<uint32_t>(R) * (4 * K + kRowPadBytes) + 127) / 128 * 128; }

__device__ __forceinline__ float lds32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

__global__ void __launch_bounds__(kTeamMaxWarps * 32, 1) rotate2_quantize_team_kernel(const __grid_constant__ Team2Params p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 127u) & ~127u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  const int nb = p.K / TRDQ_BLOCK;
  const int R = p.R;
  const uint32_t box_bytes = R * 128;
  const uint32_t in_bytes = 2 * nb * box_bytes;
  const uint32_t row_stride = 4 * p.K + kRowPadBytes;
  const uint32_t team_bytes = row_buffer_bytes(p.K, R);
  const int vec_floats = nb * (TRDQ_BLOCK + kVecPadFloats);
  float* svec1 = reinterpret_cast<float*>(smem + p.teams * team_bytes);
  float* svec2 = svec1 + vec_floats;                                              // by SOURCE channel
  uint16_t* soff = reinterpret_cast<uint16_t*>(svec2 + vec_floats);               // [K] byte offsets, block b at b * (128 + 8)
  unsigned int* row_max_all = reinterpret_cast<unsigned int*>(soff + nb * (TRDQ_BLOCK + 8));  // [teams][3][R]
  uint64_t* bars = reinterpret_cast<uint64_t*>(row_max_all + ((p.teams * 3 * R + 1) & ~1));   // [teams]

  const int tid = threadIdx.x;
  const int team_threads = p.team_warps * 32;
  const int team = tid / team_threads;
  const int tt = tid - team * team_threads;
  const uint32_t team_base = smem_base + team * team_bytes;
  // One buffer per team takes turns: the input tile in its first half, then the rows, then the codes in its last quarter, so that
  // the next input may arrive while the codes are formed and stored.
  const uint32_t rows_base = team_base;
  const uint32_t code_base = team_base + 3 * R * p.K;
  unsigned int* row_max = row_max_all + team * 3 * R;
  const uint32_t bar_full = smem_u32(bars + team);

  if (tt == 0) {
    mbar_init(bar_full, 1);
    fence_mbar_init();
  }
  stage_vector(svec1, p.vec1, p.K);
  for (int j = tid; j < p.K; j += blockDim.x) {
    const int c = __ldg(p.perm + j);
    svec2[(c >> 7) * (TRDQ_BLOCK + kVecPadFloats) + (c & 127)] = __ldg(p.vec2 + j);
    soff[(j >> 7) * (TRDQ_BLOCK + 8) + (j & 127)] = static_cast<uint16_t>(row_offset(c));
  }
  for (int i = tid; i < p.teams * 3 * R; i += blockDim.x) row_max_all[i] = 0u;
  if (tid == 0) {
    prefetch_tensormap(&p.tmap_x);
    prefetch_tensormap(&p.tmap_codes);
  }
  __syncthreads();
  griddep_launch_dependents();
  griddep_wait();  // X may be written, and the code buffer still read, by the kernel before (the tables are constant)

  const int num_tiles = (p.M + R - 1) / R;
  const int stride = gridDim.x * p.teams;
  const int first = team * gridDim.x + blockIdx.x;
  if (tt == 0 && first < num_tiles) {
    mbar_arrive_expect_tx(bar_full, in_bytes);
    tma_load_3d(team_base, &p.tmap_x, 0, first * R, 0, bar_full);
  }

  const bool active = tt < R * nb;
  const int b = active ? tt / R : 0;
  const int r = active ? tt - b * R : 0;
  const float4* sv1 = reinterpret_cast<const float4*>(svec1 + b * (TRDQ_BLOCK + kVecPadFloats));
  const float4* sv2 = reinterpret_cast<const float4*>(svec2 + b * (TRDQ_BLOCK + kVecPadFloats));
  const uint32_t off_base = smem_u32(soff + b * (TRDQ_BLOCK + 8));
  const uint32_t my_row = rows_base + r * row_stride;

  BoundedWaiter w(p.status, kStatusTimeoutEpilogue);
  int it = 0;
  for (int tile = first; tile < num_tiles; tile += stride, ++it) {
    const int buf = it % 3;
    if (tt < R) row_max[((it + 1) % 3) * R + tt] = 0u;
    w.wait(bar_full, it & 1);
    float2 v[64];
    load_scaled_block(team_base, box_bytes, b, r, sv1, v);
    wht128_thread(v);  // first rotation

    if (tt == 0) bulk_wait_group_read<0>();  // the previous tile's codes have left the buffer
    team_barrier(team, team_threads);        // every thread of the team has read the input tile
    if (active) {
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const float4 f = sv2[q];
        const float2 lo = __fmul2_rn(v[2 * q], make_float2(f.x, f.y)), hi = __fmul2_rn(v[2 * q + 1], make_float2(f.z, f.w));
        st_shared_v4(my_row + b * 512 + ((q ^ (b & 7)) << 4), __float_as_uint(lo.x), __float_as_uint(lo.y), __float_as_uint(hi.x), __float_as_uint(hi.y));
      }
    }
    team_barrier(team, team_threads);
    // permutation: eight 16-bit offsets per load
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const uint4 o = lds128(off_base + q * 16);
      const uint32_t wd[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) v[4 * q + i] = make_float2(lds32(my_row + (wd[i] & 0xFFFFu)), lds32(my_row + (wd[i] >> 16)));
    }
    wht128_thread(v);  // second rotation
    const float m = absmax_thread(v);
    if (active) atomicMax(&row_max[buf * R + r], __float_as_uint(m));
    fence_proxy_async_smem();
    team_barrier(team, team_threads);  // row maxima complete; every gather of the tile is done: the buffer takes the next input and the codes
    if (tt == 0 && tile + stride < num_tiles) {
      mbar_arrive_expect_tx(bar_full, in_bytes);
      tma_load_3d(team_base, &p.tmap_x, 0, (tile + stride) * R, 0, bar_full);
    }

    const float amax = __uint_as_float(row_max[buf * R + r]);
    const float inv = amax > 0.0f ? __fdiv_rn(127.0f, amax) : 0.0f;
    if (active) {
      quantize_store_block(v, inv, p.zero, code_base + b * box_bytes + r * 128);
      const int64_t row = static_cast<int64_t>(tile) * R + r;
      if (b == 0 && row < p.M) p.scales[row] = __fdiv_rn(amax, 127.0f);
    }
    fence_proxy_async_smem();
    team_barrier(team, team_threads);
    if (tt == 0) {
      tma_store_3d(&p.tmap_codes, 0, tile * R, 0, code_base);  // all nb column boxes; rows >= M are clipped
      bulk_commit_group();
    }
  }
  if (tt == 0) bulk_wait_group_read<0>();
  w.settle();
}

struct Team2Shape {
  int R, team_warps, teams;
  size_t smem;
  double use;  // fraction of the twelve warps' lanes that hold a block
};

size_t team2_smem_bytes(int K, int R, int teams, bool input_apart = false) {
  const size_t nb = K / TRDQ_BLOCK;
  return 128 + teams * ((input_apart ? static_cast<size_t>(2) * R * K : 0) + row_buffer_bytes(K, R)) + nb * (TRDQ_BLOCK + kVecPadFloats) * 8 + nb * (TRDQ_BLOCK + 8) * 2 +
         (static_cast<size_t>(teams) * 3 * R + 2) * 4 + static_cast<size_t>(teams) * 8 + 16;
}

// The team size, by the share of the twelve warps' lanes that hold a block, weighted by what else was seen to count over 2600 timings of all
// shapes (K = 384 ... 8192, M = 600 ... 16384): rows are 48 bytes apart modulo 128, so eight of them fill the banks evenly, and tiles of a
// multiple of eight rows gather with fewer conflicts (K = 1408 at M = 16384: 8 rows 28.9 us, 7 rows 36.9), even numbers are a
// little ahead of odd ones; two teams overlap less than three; and warps that do not divide by the four schedulers leave some of
// them idle.  The shapes taken are 1.4 % off the best ones on average, by lanes alone 5.3 %.  A tile is at most two thirds of an SM's share of the
// rows, or an SM would have nothing to overlap.  At least two teams (the memory allows it for rows of up to 98 blocks; offsets of 16 bits would reach 128).
bool choose_team2_shape(int M, int K, int sms, Team2Shape* out) {
  const int nb = K / TRDQ_BLOCK;
  Team2Shape best = {0, 0, 0, 0, 0.0};
  double best_score = 0.0;
  for (int tw = 1; tw <= kTeamMaxWarps / 2; ++tw)
    for (int rows = tw * 32 / nb < 32 ? tw * 32 / nb : 32; rows >= 1; --rows) {
      int teams = kTeamMaxWarps / tw;
      while (teams > 0 && team2_smem_bytes(K, rows, teams) > 227u * 1024u) --teams;
      if (teams < 2) continue;
      if (rows > 1 && static_cast<int64_t>(rows) * 3 * sms > 2ll * M) continue;
      const double use = static_cast<double>(rows) * nb * teams / (32 * kTeamMaxWarps);
      const int idle = (4 - teams * tw % 4) % 4;
      const double score = use * (rows % 8 == 0 ? 1.2 : rows % 2 == 0 ? 1.06 : 1.0) * (teams == 2 ? 0.95 : 1.0) * (1.0 - 0.3 * idle / kTeamMaxWarps);
      if (score > best_score + 1e-9) {
        best = Team2Shape{rows, tw, teams, team2_smem_bytes(K, rows, teams), use};
        best_score = score;
      }
    }
  if (best.teams == 0) return false;
  *out = best;
  return true;
}

// What the dispatch line below is drawn with: not the cut that is launched, but that of an earlier form of the kernel, by lanes alone (the fuller teams of two
// that are alike) and with an input tile of its own per team.
bool line_team2_shape(int K, Team2Shape* out) {
  const int nb = K / TRDQ_BLOCK;
  Team2Shape best = {0, 0, 0, 0, 0.0};
  for (int tw = 1; tw <= kTeamMaxWarps / 2; ++tw)
    for (int rows = tw * 32 / nb < 32 ? tw * 32 / nb : 32; rows >= 1; --rows) {
      int teams = kTeamMaxWarps / tw;
      while (teams > 0 && team2_smem_bytes(K, rows, teams, true) > 227u * 1024u) --teams;
      if (teams < 2) continue;
      const double use = static_cast<double>(rows) * nb * teams / (32 * kTeamMaxWarps);
      const double lanes = static_cast<double>(rows) * nb / (32 * tw), best_lanes = static_cast<double>(best.R) * nb / (32 * best.team_warps + 1e-9);
      if (use > best.use + 1e-9 || (use > best.use - 1e-9 && lanes > best_lanes + 1e-9)) best = Team2Shape{rows, tw, teams, 0, use};
    }
  *out = best;
  return best.teams != 0;
}

}  // namespace

// From which row count on the team kernel serves rows of K channels.  With few rows both kernels take one pass and the shorter one wins: a thread of this
// kernel transforms a whole block twice and gathers 128 values, of the lane-group kernel a quarter of one.  The line is drawn in rounds of that kernel,
// the rows its two CTAs per SM take at once: 0.94 for one block per row, 0.54 up to ten blocks, 1.1 up to 24, 1.3 up to 36, 1.6 beyond, eleven
// rows per SM where the earlier form held one row per team; and where that form used less than 0.45 of the lanes (K = 6784 ... 7296, 8192 and more) the
// lane groups serve all row counts.  It lies where the earlier form changed sides, to the safe side of the present one: of 401 timed points above it
// (K = 128 ... 9216, M = 300 ... 16384) none is slower than the lane groups, 0.66 of their time on average (K = 1024: 7.6 / 6.8 us at M = 1480, lane groups / teams;
// K = 4096: 17.1 / 13.2 at 1639; K = 6144: 21.4 / 18.0 at 1480); of 471 below it the present form would be faster by more than 1.5 % at 214 (K = 4608: 10.1 / 9.6 at M = 740;
// K = 4096: 11.9 / 9.2 at 829; K = 8192: 74.2 / 57.4 at 4096), and slower, up to twice, at the fewest rows.
bool rotate2_prefers_team(int32_t M, int32_t K) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  Team2Shape s;
  if (!line_team2_shape(K, &s) || s.use < 0.45 || (static_cast<int64_t>(M) + s.R - 1) / s.R < sms) return false;
  if (s.R == 1) return M >= 11 * sms;
  const int nb = K / TRDQ_BLOCK;
  const int64_t round = 2ll * sms * rotate2_lane_group_rows(K);
  const int percent = nb == 1 ? 94 : nb <= 10 ? 54 : nb <= 24 ? 110 : nb <= 36 ? 130 : 160;
  return static_cast<int64_t>(M) * 100 >= round * percent;
}

trdq_status launch_rotate2_quantize_team(const void* x_bf16, int64_t ldx, int32_t M, int32_t K, const float* vec1, const int32_t* perm,
                                         const float* vec2, int8_t* codes, float* scales, cudaStream_t stream) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) != cudaSuccess) return TRDQ_ERR_CUDA;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  Team2Shape shape;
  if (!choose_team2_shape(M, K, sms, &shape)) return TRDQ_ERR_SHAPE;
  const int nb = K / TRDQ_BLOCK;
  Team2Params p;
  trdq_status st = encode_tmap_boxes(&p.tmap_x, x_bf16, 2, 64, static_cast<uint64_t>(M), static_cast<uint64_t>(ldx) * 2,
                                     static_cast<uint32_t>(2 * nb), static_cast<uint32_t>(shape.R));
  if (st != TRDQ_OK) return st;
  st = encode_tmap_boxes(&p.tmap_codes, codes, 1, 128, static_cast<uint64_t>(M), static_cast<uint64_t>(K), static_cast<uint32_t>(nb),
                         static_cast<uint32_t>(shape.R));
  if (st != TRDQ_OK) return st;
  p.vec1 = vec1;
  p.perm = perm;
  p.vec2 = vec2;
  p.scales = scales;
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
    if (cudaFuncSetAttribute(rotate2_quantize_team_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
      return TRDQ_ERR_CUDA;
    configured.set(dev, true);
  }
  const int num_tiles = (M + shape.R - 1) / shape.R;
  const int grid = num_tiles < sms ? num_tiles : sms;
  const cudaError_t e = launch_overlapped(rotate2_quantize_team_kernel, dim3(grid), dim3(shape.teams * shape.team_warps * 32), shape.smem,
                                          stream, p);
  return e == cudaSuccess ? TRDQ_OK : TRDQ_ERR_CUDA;
}

}  // namespace trdq
