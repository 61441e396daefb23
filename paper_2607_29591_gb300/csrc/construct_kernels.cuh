// Construction kernels (Alg. 1) -- token scoring, ranking, Lloyd residual
// entries, validation proxy and packing.  Included once, by construct.cu.
#pragma once
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <climits>
#include <cstdint>

#include "device_utils.cuh"
#include "internal.h"
#include "mma_tile.cuh"

namespace reskv {
namespace build {

namespace cg = cooperative_groups;

constexpr int kTile = 128;          // tokens per tile
constexpr int kThreads = 256;       // 8 warps

// ---------------------------------------------------------------------------
// Shared-memory tiles
// ---------------------------------------------------------------------------

constexpr int kAsgRowBytes = kHeadDim * 2;  // one bf16 row of 128 dims

// byte offset of 16-byte chunk `ch` of row `row` in a [rows][256 B] bf16 tile;
// chunks XOR-swizzled by row so that ldmatrix reads of 8 rows are conflict free
__device__ __forceinline__ uint32_t asg_swz(int row, int ch) {
  return uint32_t(row) * kAsgRowBytes + uint32_t((ch ^ (row & 7)) << 4);
}

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(src_bytes)
               : "memory");
}

// the same for 8 bytes on an 8-byte boundary
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Stage the bf16 keys of tokens tok0..tok0+127 as a swizzled [128][256 B]
// tile (zeros past s); the copies complete at the caller's wait.
__device__ __forceinline__ void stage_key_tile(uint32_t ks_s, const __nv_bfloat16* Ku, int64_t s,
                                               int64_t tok0) {
  for (int idx = threadIdx.x; idx < kTile * 16; idx += blockDim.x) {
    const int row = idx >> 4, ch = idx & 15;
    const bool in = tok0 + row < s;
    cp_async16(ks_s + asg_swz(row, ch), Ku + (in ? (tok0 + row) * kHeadDim : 0) + 8 * ch,
               in ? 16u : 0u);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Token scores (App. B.2 SnapKV rule; Alg. 1)
// ---------------------------------------------------------------------------

struct ObsArgs {
  const __nv_bfloat16* K;      // layer keys [UL, s, d]
  const __nv_bfloat16* Qobs;   // layer observation queries [UL*G, n_obs, d]
  int64_t s;
  int32_t G, n_obs, n_rows;    // n_rows = G * n_fit, row = g * n_fit + t
  int32_t n_fit;
  int32_t ntiles;
  uint4* qfrag;                // [UL, blocks of 16 rows, 8, 32] the fit rows as A fragments
  float2* tile_stats;          // [UL, n_rows, ntiles] (max, sum) per tile, log2 domain
  float2* row_stats;           // [UL, n_rows] (max, 1/sum)
  float* A;                    // [UL, s] attention summed over fit rows, averaged over G
};

// Logits of the fit rows against tiles of 128 keys on the tensor cores
// (mma.sync m16n8k16): the queries are the A operand, 16 rows to a block, the
// keys the B operand from the swizzled tile.  Products of the bf16 rows and keys
// are exact, accumulated in fp32, then scaled by log2(e)/sqrt(d) (the logits in
// log2 units).  The accumulator of n-tile nt holds rows g (entries 0, 1) and
// g + 8 (entries 2, 3) at tokens 8 nt + 2 t4 (+1), with g = lane / 4,
// t4 = lane % 4.
//
// What bounds it: reading fragments from shared memory and L1 (65 and 81 % of
// the data pipe's wavefronts in the two passes, the tensor pipe 32 and 26 %, with
// 16 rows per fragment of keys and the queries gathered row by row for every
// tile).  So a warp takes two blocks of rows (32 rows) per fragment of keys, and
// the queries come as whole fragments, laid out once per layer (k_obs_frag).  The
// block has as many warps as there are row pairs to share evenly, and several
// blocks per SM cover each other's loads.  64 units of 32K keys, 96 rows: passes
// 361 + 472 us -> 204 + 252; 32 units of 128K keys, 384 rows: 2039 + 2579 ->
// 1375 + 1273 (the tensor pipe, busy for about half of that, and the issue of the
// exponentials between the products bound it now; the second pass, at 168
// registers, spills 228 bytes a thread and reads 396 back: two blocks per SM
// without the spills took 350 us where this takes 252).
__global__ void k_obs_frag(ObsArgs p) {          // grid (blocks of rows, UL), 256 threads
  const int rb = blockIdx.x, ul = blockIdx.y;
  const int ks = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  auto row = [&](int r) -> const uint32_t* {
    if (r >= p.n_rows) return nullptr;
    const int h = r / p.n_fit, t = r % p.n_fit;
    return reinterpret_cast<const uint32_t*>(p.Qobs + ((int64_t(ul) * p.G + h) * p.n_obs + t) * kHeadDim) + 8 * ks + t4;
  };
  const uint32_t *q0 = row(rb * 16 + g), *q1 = row(rb * 16 + g + 8);
  p.qfrag[((int64_t(ul) * gridDim.x + rb) * 8 + ks) * 32 + lane] =
      make_uint4(q0 ? __ldg(q0) : 0u, q1 ? __ldg(q1) : 0u, q0 ? __ldg(q0 + 4) : 0u, q1 ? __ldg(q1 + 4) : 0u);
}

// the A fragments of row blocks rb and rb + 1 (zeros past the last block)
__device__ __forceinline__ void obs_load_a(const ObsArgs& p, int ul, int rb, int nrb, int lane, uint4 (&A)[2][8]) {
  const uint4* f = p.qfrag + (int64_t(ul) * nrb + rb) * 256 + lane;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) A[0][ks] = __ldg(f + 32 * ks);
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) A[1][ks] = rb + 1 < nrb ? __ldg(f + 256 + 32 * ks) : make_uint4(0, 0, 0, 0);
}

// logits of the (one or) two row blocks against tokens tk .. tk + 16 NP - 1 of the tile
template <int NP>
__device__ __forceinline__ void obs_logits(uint32_t ks_s, int tk, int lane, const uint4 (&A)[2][8], bool two,
                                           float (&S)[2][2 * NP][4]) {
  const int mi = lane >> 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int nt = 0; nt < 2 * NP; ++nt) S[i][nt][0] = S[i][nt][1] = S[i][nt][2] = S[i][nt][3] = 0.f;
  const int trow = tk + (mi >> 1) * 8 + (lane & 7);
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
#pragma unroll
    for (int np = 0; np < NP; ++np) {
      uint32_t b0, b1, b2, b3;
      ldsm_x4(ks_s + asg_swz(trow + 16 * np, 2 * ks + (mi & 1)), b0, b1, b2, b3);
      mma16816(S[0][2 * np], A[0][ks].x, A[0][ks].y, A[0][ks].z, A[0][ks].w, b0, b1);
      mma16816(S[0][2 * np + 1], A[0][ks].x, A[0][ks].y, A[0][ks].z, A[0][ks].w, b2, b3);
      if (two) {
        mma16816(S[1][2 * np], A[1][ks].x, A[1][ks].y, A[1][ks].z, A[1][ks].w, b0, b1);
        mma16816(S[1][2 * np + 1], A[1][ks].x, A[1][ks].y, A[1][ks].z, A[1][ks].w, b2, b3);
      }
    }
  const float scale = kLog2e * rsqrtf(float(kHeadDim));
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int nt = 0; nt < 2 * NP; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) S[i][nt][e] *= scale;
}

// Warps of a block of the first pass: one per pair of row blocks where there are
// few, else 4, or 3 where that leaves fewer idle in the last round.
__host__ inline int obs_warps1(int n_rows) {
  const int pairs = ((n_rows + 15) / 16 + 1) / 2;
  if (pairs <= 3) return pairs;
  return (pairs + 2) / 3 * 3 < (pairs + 3) / 4 * 4 ? 3 : 4;
}
// of the second: its items are (pair of partial sums, half of the tile)
__host__ inline int obs_warps2(int n_rows) {
  const int pairs = (std::min((n_rows + 15) / 16, 8) + 1) / 2;
  return pairs <= 2 ? 2 * pairs : pairs;
}

// (max, sum) of one row's 16 logits of this lane and its three neighbours'
// (64 tokens), folded into the row's; n tokens of the half exist
template <bool ragged>
__device__ __forceinline__ void obs_fold(const float (&S)[8][4], int a, int t4, int n, float& M, float& L) {
  float mx = -INFINITY;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int c = 0; c < 2; ++c)
      if (!ragged || 8 * nt + 2 * t4 + c < n) mx = fmaxf(mx, S[nt][2 * a + c]);
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  float sum = 0.f;
  if (mx != -INFINITY) {
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (!ragged || 8 * nt + 2 * t4 + c < n) sum += exp2f(S[nt][2 * a + c] - mx);
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  if (mx != -INFINITY) {
    const float nm = fmaxf(M, mx);
    L = L * exp2f(M - nm) + sum * exp2f(mx - nm);
    M = nm;
  }
}

// Pass 1: per (row, tile) max and sum of 2^{a log2e} over the tile's tokens.
__global__ void __launch_bounds__(128, 3) k_obs_pass1(ObsArgs p) {
  extern __shared__ __align__(128) uint8_t obs_raw[];
  const int tile = blockIdx.x, ul = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int64_t tok0 = int64_t(tile) * kTile;
  const uint32_t ks_s = smem_u32(obs_raw);
  stage_key_tile(ks_s, p.K + int64_t(ul) * p.s * kHeadDim, p.s, tok0);
  const int nrb = (p.n_rows + 15) / 16, n_tok = int(min(int64_t(kTile), p.s - tok0));
  uint4 A[2][8];
  obs_load_a(p, ul, 2 * w, nrb, lane, A);        // (every warp has a pair)
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (int rb = 2 * w; rb < nrb;) {
    const bool two = rb + 1 < nrb;
    float M[2][2], L[2][2];                      // rows g, g + 8 of the two blocks
#pragma unroll
    for (int i = 0; i < 2; ++i) M[i][0] = M[i][1] = -INFINITY, L[i][0] = L[i][1] = 0.f;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      float S[2][8][4];
      obs_logits<4>(ks_s, 64 * h, lane, A, two, S);
      const int n = n_tok - 64 * h;
      if (n >= 64) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int a = 0; a < 2; ++a) obs_fold<false>(S[i], a, t4, n, M[i][a], L[i][a]);
      } else {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int a = 0; a < 2; ++a) obs_fold<true>(S[i], a, t4, n, M[i][a], L[i][a]);
      }
    }
    if (t4 == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int row = (rb + i) * 16 + g + 8 * a;
          if (row < p.n_rows)
            p.tile_stats[(int64_t(ul) * p.n_rows + row) * p.ntiles + tile] = make_float2(M[i][a], L[i][a]);
        }
    }
    rb += 2 * (blockDim.x >> 5);
    if (rb < nrb) obs_load_a(p, ul, rb, nrb, lane, A);
  }
}

// Row statistics over all tiles: the sums in tile order, one chain of fused
// multiply-adds per row.  32 rows per block of 256 threads: the maxima and the
// exponentials take eight threads a row, the chains a lane each, one chunk of
// tiles behind.  Latency bound (the chain: 4 cycles a tile); 3072 rows of 256
// tiles: 9 us, 99 with the loads and exponentials in the chain too.
constexpr int kStatChunk = 64;

__global__ void __launch_bounds__(256) k_obs_rowstats(ObsArgs p, int UL) {
  __shared__ float2 term[2][32][kStatChunk + 1];
  const int64_t n = int64_t(UL) * p.n_rows, row0 = int64_t(blockIdx.x) * 32;
  const int rl = threadIdx.x >> 3, sub = threadIdx.x & 7, lane = threadIdx.x & 31;
  const bool in = row0 + rl < n;
  const float2* t = p.tile_stats + (row0 + rl) * p.ntiles;
  float mx = -INFINITY;
  if (in)
    for (int k = sub; k < p.ntiles; k += 8) mx = fmaxf(mx, t[k].x);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int nch = (p.ntiles + kStatChunk - 1) / kStatChunk;
  float sum = 0.f;
  for (int c = 0; c <= nch; ++c) {
    if (c < nch && in) {
#pragma unroll
      for (int j = 0; j < kStatChunk / 8; ++j) {
        const int k = c * kStatChunk + sub + 8 * j;
        const float2 v = k < p.ntiles ? t[k] : make_float2(0.f, 0.f);
        term[c & 1][rl][sub + 8 * j] = v.y > 0.f ? make_float2(v.y, exp2f(v.x - mx)) : make_float2(0.f, 0.f);
      }
    }
    if (c > 0 && threadIdx.x < 32) {
      const float2* v = term[(c - 1) & 1][lane];
#pragma unroll 16
      for (int k = 0; k < kStatChunk; ++k) sum += v[k].x * v[k].y;
    }
    __syncthreads();
  }
  // the row's maximum lies with its eight threads, its sum with lane `row` of warp 0
  float* m_s = reinterpret_cast<float*>(term);
  if (sub == 0) m_s[rl] = mx;
  __syncthreads();
  if (threadIdx.x < 32 && row0 + lane < n) p.row_stats[row0 + lane] = make_float2(m_s[lane], 1.0f / sum);
}

// the softmax weights of two row blocks, added to this lane's column sums of the
// 64 tokens from tk on; all: every row has a finite positive sum
template <bool all>
__device__ __forceinline__ void obs_columns(uint32_t ks_s, int tk, int lane, const uint4 (&A)[2][8], bool two,
                                            const float2 (&st)[2][2], float (&col)[2][8][2]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {                  // 32 tokens at a time
    float S[2][4][4];
    obs_logits<2>(ks_s, tk + 32 * q, lane, A, two, S);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int a = 0; a < 2; ++a)
            if (all || st[i][a].y > 0.f) col[i][4 * q + nt][c] += exp2f(S[i][nt][2 * a + c] - st[i][a].x) * st[i][a].y;
  }
}

// Pass 2: A_p = (1/G) sum over fit rows of the softmax weight of token p.  The
// sums are formed apart for the row blocks congruent mod 8, in ascending order,
// and added in the order of the remainders: a warp takes two remainders and half
// of the tile's tokens.
__global__ void __launch_bounds__(128, 3) k_obs_pass2(ObsArgs p) {
  extern __shared__ __align__(128) uint8_t obs_raw[];
  float* red = reinterpret_cast<float*>(obs_raw + kTile * kAsgRowBytes);   // [8 remainders][128 tokens]
  const int tile = blockIdx.x, ul = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int64_t tok0 = int64_t(tile) * kTile;
  const uint32_t ks_s = smem_u32(obs_raw);
  stage_key_tile(ks_s, p.K + int64_t(ul) * p.s * kHeadDim, p.s, tok0);
  const int nrb = (p.n_rows + 15) / 16, n_rem = min(nrb, 8), pairs = (n_rem + 1) / 2;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (int it = w; it < 2 * pairs; it += blockDim.x >> 5) {
    // with four pairs: the first two, which may have a block of rows more, share
    // the first round
    const int pr = pairs == 4 ? 2 * (it >> 2) + (it & 1) : it % pairs, h = pairs == 4 ? (it >> 1) & 1 : it / pairs;
    float col[2][8][2];                          // this lane's column sums
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) col[i][nt][0] = col[i][nt][1] = 0.f;
#pragma unroll 1
    for (int rb = 2 * pr; rb < nrb; rb += 8) {
      const bool two = rb + 1 < nrb;
      uint4 A[2][8];
      obs_load_a(p, ul, rb, nrb, lane, A);
      float2 st[2][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int row = (rb + i) * 16 + g + 8 * a;
          st[i][a] = row < p.n_rows ? p.row_stats[int64_t(ul) * p.n_rows + row] : make_float2(0.f, 0.f);
        }
      const bool all = __all_sync(0xffffffffu, st[0][0].y > 0.f && st[0][1].y > 0.f && st[1][0].y > 0.f && st[1][1].y > 0.f);
      if (all) {
        obs_columns<true>(ks_s, 64 * h, lane, A, true, st, col);
      } else {                                   // rows past the last, or without a finite sum
        obs_columns<false>(ks_s, 64 * h, lane, A, two, st, col);
      }
    }
    // sum over the eight row groups of the warp (the remainders are summed below)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float v = col[i][nt][c];
          v += __shfl_xor_sync(0xffffffffu, v, 4);
          v += __shfl_xor_sync(0xffffffffu, v, 8);
          v += __shfl_xor_sync(0xffffffffu, v, 16);
          if (g == 0) red[(2 * pr + i) * kTile + 64 * h + 8 * nt + 2 * t4 + c] = v;
        }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kTile; i += blockDim.x) {
    float a = 0.f;
    for (int rem = 0; rem < n_rem; ++rem) a += red[rem * kTile + i];
    const int64_t tok = tok0 + i;
    if (tok < p.s) p.A[int64_t(ul) * p.s + tok] = a / float(p.G);
  }
}

// Zero-padded average pooling of width `pool` (odd), summed in fp64 in ascending
// order; inv = RN(1 / pool).  Bound by fp64, scarce on this part: a thread takes
// four positions, so a value is converted once for them, and divides by
// Markstein's correction (q0 = RN(a inv), r = a - q0 pool exactly, q = RN(q0 + r inv):
// with an odd divisor a / pool lies at least 1 / (2 pool) ulp from a rounding
// boundary, far more than the correction is off by).  4.2M positions, width 7: 107
// us, 150 with a conversion per term and a division.
__global__ void __launch_bounds__(256) k_pool(const float* __restrict__ A, double* __restrict__ scores, int64_t s, int UL,
                                              int pool, double inv) {
  const int64_t runs = (s + 3) / 4, i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(UL) * runs) return;
  const int64_t ul = i / runs, p0 = i % runs * 4;
  const float* Au = A + ul * s;
  const int half = pool / 2;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int j = -half; j < half + 4; ++j) {       // value p0 + j belongs to positions p0 + j - half .. p0 + j + half
    const int64_t q = p0 + j;
    if (q < 0 || q >= s) continue;
    const double v = double(__ldg(Au + q));
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (j >= k - half && j <= k + half) acc[k] += v;
  }
  const double n = double(pool);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double q0 = acc[k] * inv;
    if (p0 + k < s) scores[ul * s + p0 + k] = fma(fma(-q0, n, acc[k]), inv, q0);
  }
}

// Query-free score ||k_p||^2 (a build choice; the paper defines none): the
// exact sum of the squares, rounded once to the nearest fp64 value (ties to
// even), so it does not depend on any summation order.
//
// A bf16 value is M 2^e with an integer M < 2^8 (M = 128 + mantissa field for
// normal values, the mantissa field for subnormals), so its square is
// M^2 2^t with M^2 < 2^16 and t = 2e even, t in [-266, 242].  The common row
// (k_key_norms): every nonzero value lies within 20 binades of the largest, so
// all values are integers below 2^28 in units of the lowest of those binades,
// their squares sum below 2^63 in 64-bit integers, one multiply-add each, and
// one conversion rounds the sum (within 13 binades a float addition forms the
// integer, else a shift).  Otherwise a warp takes the row
// (keynorm_row): with tmax the largest t of the row's nonzero squares, every
// square with t >= tmax - 104 is an exact integer multiple of 2^(tmax - 104)
// below 2^120, and 128 of them sum below 2^127: it adds them as 128-bit
// integers.  A row with a nonzero square below that window (its values span
// more than 52 binades) goes to an exact 576-bit accumulator in one lane.

using u128 = unsigned __int128;

// Correctly rounded fp64 value of a 2^base, a > 0; `sticky`: a positive
// amount below a's last bit is to be added as well.
__device__ inline double round_u128(u128 a, int base, bool sticky) {
  const uint64_t hi = uint64_t(a >> 64), lo = uint64_t(a);
  const int p = hi ? 127 - __clzll((long long)hi) : 63 - __clzll((long long)lo);
  if (p <= 52) return ldexp(double(lo), base);            // exact (sticky never set here)
  const int sh = p - 52;
  uint64_t mant = uint64_t(a >> sh);
  const u128 one = 1;
  const u128 rem = a & ((one << sh) - 1), half = one << (sh - 1);
  if (rem > half || (rem == half && (sticky || (mant & 1u)))) ++mant;
  return ldexp(double(mant), base + sh);
}

// The square of one bf16 value as (M^2, t); M^2 = 0 for zero.
__device__ inline void bf16_square(uint32_t b, uint32_t& m2, int& t, bool& finite) {
  const uint32_t ef = (b >> 7) & 0xffu, mf = b & 0x7fu;
  const uint32_t M = ef ? 128u + mf : mf;
  m2 = M * M;
  t = 2 * (int(ef ? ef : 1u) - 134);
  finite = ef != 0xffu;
}

// Exact sum of a row's squares in 32-bit digits (bit q = t + 266 of the sum
// in digit q / 32), then the correctly rounded fp64 value.  One thread.
__device__ double keynorm_wide(const __nv_bfloat16* rowp) {
  const uint16_t* bits = reinterpret_cast<const uint16_t*>(rowp);
  uint64_t dig[18];
#pragma unroll
  for (int j = 0; j < 18; ++j) dig[j] = 0;
  for (int i = 0; i < kHeadDim; ++i) {
    uint32_t m2;
    int t;
    bool fin;
    bf16_square(bits[i], m2, t, fin);
    if (!m2) continue;
    const int q = t + 266;
    const uint64_t v = uint64_t(m2) << (q & 31);
    dig[q >> 5] += v & 0xffffffffu;
    dig[(q >> 5) + 1] += v >> 32;
  }
  for (int j = 0; j < 17; ++j) {
    dig[j + 1] += dig[j] >> 32;
    dig[j] &= 0xffffffffu;
  }
  int top = 17;
  while (top > 0 && dig[top] == 0) --top;
  u128 a = 0;
  for (int j = top; j > top - 4; --j) a = (a << 32) | (j >= 0 ? dig[j] : 0u);
  bool sticky = false;
  for (int j = 0; j < top - 3; ++j) sticky |= dig[j] != 0;
  return a ? round_u128(a, (top - 3) * 32 - 266, sticky) : 0.0;
}

// The exact score of any row, by a whole warp; the result is valid in lane 0.
__device__ __noinline__ double keynorm_row(const __nv_bfloat16* rowp, int lane) {
  const uint2 w = __ldg(reinterpret_cast<const uint2*>(rowp) + lane);
  const uint32_t b[4] = {w.x & 0xffffu, w.x >> 16, w.y & 0xffffu, w.y >> 16};
  uint32_t m2[4];
  int t[4];
  bool finite = true;
  int tmax = INT_MIN;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    bool f;
    bf16_square(b[j], m2[j], t[j], f);
    finite &= f;
    if (m2[j]) tmax = max(tmax, t[j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tmax = max(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
  if (!__all_sync(0xffffffffu, finite)) {                 // inf or NaN: the fp64 sum is too
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double x = double(__uint_as_float(b[j] << 16));
      acc += x * x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
  }
  if (tmax == INT_MIN) return 0.0;                        // every value is zero
  bool wide = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) wide |= m2[j] != 0 && t[j] < tmax - 104;
  if (__any_sync(0xffffffffu, wide)) return lane == 0 ? keynorm_wide(rowp) : 0.0;
  u128 a = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (m2[j]) a += u128(m2[j]) << (t[j] - tmax + 104);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t hi = __shfl_xor_sync(0xffffffffu, uint64_t(a >> 64), o);
    const uint64_t lo = __shfl_xor_sync(0xffffffffu, uint64_t(a), o);
    a += (u128(hi) << 64) | lo;
  }
  return lane == 0 ? round_u128(a, tmax - 104, false) : 0.0;
}

// the greater of two signed 16-bit halves each
__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// 128 fp32 products summed in any order stay within 130 u of the sum, the root
// and the product within 2 u each; what underflows is below 255 * 2^-150, its root
// far below kNormLost, which the caller adds (2^-50: see k_lloyd_assign's bound)
constexpr float kNormLost = 0x1p-50f;
__device__ __forceinline__ float norm_bound(float sum) { return sqrtf(sum) * (1.0f + 140.0f * 5.9604645e-8f); }

// Per key row, in one read of the keys: with kScore the query-free score, and
// (knorm not NULL) an upper bound of ||k|| for the Lloyd assignment's rounding
// bound.  n_rows rows of 256 bytes.
//
// A warp takes 32 rows, four at a time with eight lanes each (two 16-byte loads
// a lane, four rows' worth in flight; keys on an 8-byte boundary take 8-byte
// loads), and every lane keeps the sum of one row, so the conversion and the root
// are done once for 32 rows.  The bound alone runs at the DRAM rate (2.1M rows: 77
// us, 194 with a warp per row); with the scores the integer sums issue for longer
// than the loads take (8.4M rows, 2.1 GB: 505 us for both, 645 with shifts for
// every row, 2883 + 768 with a warp per row and 128-bit sums).
template <bool kScore>
__global__ void __launch_bounds__(256) k_key_norms(const __nv_bfloat16* __restrict__ K, double* __restrict__ scores,
                                                   float* __restrict__ knorm, int64_t n_rows) {
  const int64_t base = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * 32;
  if (base >= n_rows) return;                             // whole warps leave together
  const int lane = threadIdx.x & 31, q = lane >> 3, c = lane & 7;
  const bool wide = (reinterpret_cast<uintptr_t>(K) & 15u) == 0;
  const int64_t mine = base + 4 * c + q;                  // the row whose sum this lane keeps
  uint64_t sum = 0;                                       // kScore: in units of 2^(2 (e0 - 134))
  float fsum = 0.f;
  int e0 = 0;                                             // 0: not a common row
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint4 w[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t row = base + 4 * (4 * half + i) + q;
      w[i][0] = w[i][1] = make_uint4(0, 0, 0, 0);
      if (row < n_rows) {
        const __nv_bfloat16* src = K + row * kHeadDim + 8 * c;
        if (wide) {
          w[i][0] = __ldg(reinterpret_cast<const uint4*>(src));
          w[i][1] = __ldg(reinterpret_cast<const uint4*>(src) + 8);
        } else {
          const uint2* s8 = reinterpret_cast<const uint2*>(src);
          const uint2 a = __ldg(s8), b = __ldg(s8 + 1), d = __ldg(s8 + 16), e = __ldg(s8 + 17);
          w[i][0] = make_uint4(a.x, a.y, b.x, b.y);
          w[i][1] = make_uint4(d.x, d.y, e.x, e.y);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t x[8] = {w[i][0].x, w[i][0].y, w[i][0].z, w[i][0].w,
                             w[i][1].x, w[i][1].y, w[i][1].z, w[i][1].w};
      if constexpr (kScore) {
        // u: a value's bits without the sign.  The largest u, and the largest
        // 2^15 - u of the nonzero values (a zero gives -2^15)
        uint32_t big = 0, small = 0x80008000u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          big = max_s16x2(big, x[j] & 0x7fff7fffu);
          small = max_s16x2(small, ~((x[j] | 0x80008000u) - 0x00010001u));
        }
        uint32_t mm = max_s16x2(__byte_perm(big, small, 0x5410), __byte_perm(big, small, 0x7632));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) mm = max_s16x2(mm, __shfl_xor_sync(0xffffffffu, mm, o));
        const int emax = int(mm & 0xffffu) >> 7, umin = 0x8000 - (int(mm) >> 16);
        // 13 binades (four rows of normally distributed values nearly always):
        // a float addition of 1.5 x 2^23 units leaves M in the low bits
        const bool near = emax >= 14 && emax <= 251 && umin >= ((emax - 13) << 7);
        const bool all_near = __all_sync(0xffffffffu, near);
        const int elow = all_near ? emax - 13 : emax - 20;
        uint64_t s64 = 0;
        if (all_near) {
          const uint32_t cb = (uint32_t(elow + 16) << 23) | 0x400000u;
          const float2 c2 = make_float2(__uint_as_float(cb), __uint_as_float(cb));
          long long acc = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float2 y = fadd2(bf16x2_to_float2(x[j]), c2);
            const int m0 = int(__float_as_uint(y.x) - cb), m1 = int(__float_as_uint(y.y) - cb);
            acc += (long long)m0 * m0;
            acc += (long long)m1 * m1;
          }
          s64 = uint64_t(acc);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int hw = 0; hw < 2; ++hw) {
              const uint32_t u = hw ? x[j] >> 16 : x[j];
              const int e = int((u >> 7) & 0xffu);
              // 2^(e - elow) M: zero (all bits shifted out) below elow
              uint32_t m;
              asm("shl.b32 %0, %1, %2;" : "=r"(m) : "r"((u & 0x7fu) | 0x80u), "r"(e - elow));
              s64 += uint64_t(m) * m;
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s64 += __shfl_xor_sync(0xffffffffu, s64, o);
        if (c == 4 * half + i) {
          sum = s64;
          e0 = elow >= 1 && emax != 0xff && umin >= (elow << 7) ? elow : 0;
        }
      } else {
        float f = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float2 v = bf16x2_to_float2(x[j]);
          f = fmaf(v.x, v.x, fmaf(v.y, v.y, f));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
        if (c == 4 * half + i) fsum = f;
      }
    }
  }
  if constexpr (!kScore) {
    if (mine < n_rows) knorm[mine] = norm_bound(fsum) + kNormLost;
  } else {
    if (mine < n_rows && e0) {
      scores[mine] = __ull2double_rn(sum) * __hiloint2double((1023 + 2 * (e0 - 134)) << 20, 0);
      if (knorm) {
        const int E = e0 - 134;
        const float unit = __uint_as_float(E >= -126 ? uint32_t(E + 127) << 23 : 1u << (E + 149));
        const float nrm = __fmul_ru(norm_bound(__ull2float_ru(sum)), unit) + kNormLost;
        knorm[mine] = nrm < 1.8446744e19f ? nrm : INFINITY;        // as the fp32 sum: beyond 2^64 no bound
      }
    }
    uint32_t rest = __ballot_sync(0xffffffffu, mine < n_rows && e0 == 0);
    while (rest) {                                        // the other rows, one by one
      const int l = __ffs(rest) - 1;
      rest &= rest - 1;
      const int64_t row = base + 4 * (l & 7) + (l >> 3);
      const double sc = keynorm_row(K + row * kHeadDim, lane);
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(K + row * kHeadDim) + lane);
      const float2 a = bf16x2_to_float2(v.x), b = bf16x2_to_float2(v.y);
      const float f = warp_sum(fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(b.x, b.x, b.y * b.y))));
      if (lane == 0) {
        scores[row] = sc;
        if (knorm) knorm[row] = norm_bound(f) + kNormLost;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Ranking of S \ P (Sec. 5.2, Eq. main_selection): the top n_top positions by
// score, highest first, ties to the lower position.  One thread-block cluster
// per unit, its CTAs on equal runs of positions: a radix select of the n_top-th
// largest key by 11-bit digits, an order-preserving compaction of the selected
// positions into rank 0's shared memory, and a bitonic sort there.
//
// What bounds it: the latency of few CTAs.  A layer of 8 to 64 units leaves most
// of the SMs idle with one CTA each, so a unit gets as many CTAs as the SMs allow
// (at most 8); usually three digits decide (a digit's bin that holds exactly the
// keys still wanted ends the select); sort steps over less than 32 elements are
// shuffles.  64 units of 32K keys, n_top = 960: 50 us, 171 with one CTA each,
// eight 8-bit digits and a barrier per sort step.
// ---------------------------------------------------------------------------

constexpr int kTopThreads = 1024;
constexpr int kTopMax = 8192;

struct TopArgs {
  const double* scores;   // [UL, s]
  int64_t s;
  int32_t recent;         // |P|
  int32_t n_top;          // entries to rank
  int32_t* top;           // [UL, n_top] positions in rank order
  int32_t* rank_pos;      // [UL, s]: rank, INT_MAX (never main) or -1 (protected)
  uint32_t* status;
  const int32_t* budgets; // [UL] per-unit budgets (rank min(b_u, s) - |P| each,
                          // at stride n_top), or NULL: rank n_top for every unit
};

// Budget of unit ul of the layer: its own, or the shared one.
__device__ __forceinline__ int64_t unit_budget(const int32_t* budgets, int ul, int64_t b) {
  return budgets ? int64_t(budgets[ul]) : b;
}

__device__ __forceinline__ uint64_t score_key(double v) {
  // non-negative doubles order like their bit patterns; clamp -0 and negatives to 0
  return v > 0.0 ? static_cast<uint64_t>(__double_as_longlong(v)) : 0ull;
}

__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  if (w == 0) {
    int ws = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, ws, o);
      if (lane >= o) ws += y;
    }
    if (lane < nw) warp_sums[lane] = ws;
  }
  __syncthreads();
  const int excl = x - v + (w > 0 ? warp_sums[w - 1] : 0);
  if (total) *total = warp_sums[nw - 1];
  __syncthreads();
  return excl;
}

constexpr int kSelDigit = 11;                  // bits of a radix-select digit
constexpr int kSelBins = 1 << kSelDigit;
static_assert(kSelBins == 2 * kTopThreads, "the digit search takes two bins per thread");

// What a select has decided: keys with (key & mask) > prefix are taken, and of
// those with (key & mask) == prefix the first `rem`.
struct SelState {
  uint64_t prefix, mask;
  int64_t rem;
};

// The K largest keys (K >= 1, at most the number of keys) of the cluster.
// each(f) calls f(key) for every key of this CTA.
template <typename Each>
__device__ SelState cluster_select(cg::cluster_group& cl, int64_t K, int* hist, int* warp_sums, int64_t* bcast,
                                   Each&& each) {
  SelState st{0, 0, K};
  for (int shift = 64 - kSelDigit;; shift = shift > kSelDigit ? shift - kSelDigit : 0) {
    hist[2 * threadIdx.x] = hist[2 * threadIdx.x + 1] = 0;
    __syncthreads();
    each([&](uint64_t key) {
      if ((key & st.mask) == st.prefix) atomicAdd(&hist[(key >> shift) & (kSelBins - 1)], 1);
    });
    cl.sync();
    // two bins per thread, the largest digits first: the digit of the K-th key
    const int d1 = kSelBins - 1 - 2 * int(threadIdx.x), d0 = d1 - 1;
    int h1 = 0, h0 = 0;
    for (unsigned r = 0; r < cl.num_blocks(); ++r) {
      const int* h = cl.map_shared_rank(hist, r);
      h1 += h[d1];
      h0 += h[d0];
    }
    const int above = block_exclusive_scan(h1 + h0, warp_sums, nullptr);
    if (above < st.rem && st.rem <= int64_t(above) + h1 + h0) {
      const bool hi = st.rem <= int64_t(above) + h1;
      bcast[0] = hi ? d1 : d0;
      bcast[1] = st.rem - above - (hi ? 0 : h1);
      bcast[2] = hi ? h1 : h0;
    }
    cl.sync();                       // bcast is there, and no CTA reads this one's counts any more
    // (the last digit overlaps the one before where 64 is not a multiple of
    // the width; its decided bits are the same in every key left)
    st.prefix |= uint64_t(bcast[0]) << shift;
    st.mask |= uint64_t(kSelBins - 1) << shift;
    st.rem = bcast[1];
    if (shift == 0 || bcast[2] == st.rem) return st;
    __syncthreads();                 // every thread has read bcast
  }
}

// Whether element (ka, ia) comes after (kb, ib): smaller key, or the larger
// position of equal keys.
__device__ __forceinline__ bool sort_after(uint64_t ka, int32_t ia, uint64_t kb, int32_t ib) {
  return ka < kb || (ka == kb && ia > ib);
}

// Bitonic sort by (key descending, position ascending) of E * kTopThreads
// elements; thread t holds elements t + kTopThreads q.  Steps over less than a
// warp are shuffles, over less than the CTA exchanges through shared memory
// (skey, sidx), and over more swaps between the thread's own elements.
template <int E>
__device__ void topk_sort(uint64_t (&k)[E], int32_t (&x)[E], uint64_t* skey, int32_t* sidx) {
  const int t = threadIdx.x;
  for (int size = 2; size <= E * kTopThreads; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= kTopThreads) {
        const int qs = stride / kTopThreads;
#pragma unroll
        for (int q = 0; q < E; ++q) {
          if ((q & qs) == 0 && q + qs < E) {
#pragma unroll
            for (int o = 0; o < E; ++o) {      // o = q + qs, with a constant index
              if (o == q + qs) {
                const bool up = ((t + kTopThreads * q) & size) == 0;
                if (sort_after(k[q], x[q], k[o], x[o]) == up) {
                  const uint64_t tk = k[q];
                  const int32_t tx = x[q];
                  k[q] = k[o];
                  x[q] = x[o];
                  k[o] = tk;
                  x[o] = tx;
                }
              }
            }
          }
        }
        continue;
      }
      if (stride >= 32) {
#pragma unroll
        for (int q = 0; q < E; ++q) {
          skey[t + kTopThreads * q] = k[q];
          sidx[t + kTopThreads * q] = x[q];
        }
        __syncthreads();
      }
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const int e = t + kTopThreads * q;
        uint64_t ok;
        int32_t ox;
        if (stride >= 32) {
          ok = skey[e ^ stride];
          ox = sidx[e ^ stride];
        } else {
          ok = __shfl_xor_sync(0xffffffffu, k[q], stride);
          ox = __shfl_xor_sync(0xffffffffu, x[q], stride);
        }
        // the lower element of an ascending pair keeps the one that comes first
        const bool first = ((e & stride) == 0) == ((e & size) == 0);
        if (sort_after(k[q], x[q], ok, ox) == first) {
          k[q] = ok;
          x[q] = ox;
        }
      }
      if (stride >= 32) __syncthreads();
    }
  }
}

template <int E>
__device__ void topk_rank(const TopArgs& p, int ul, int K, uint64_t* skey, int32_t* sidx) {
  uint64_t k[E];
  int32_t x[E];
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int e = int(threadIdx.x) + kTopThreads * q;
    k[q] = e < K ? skey[e] : 0ull;
    x[q] = e < K ? sidx[e] : INT_MAX;          // padding sorts last
  }
  __syncthreads();
  topk_sort<E>(k, x, skey, sidx);
  int32_t* rp = p.rank_pos + int64_t(ul) * p.s;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int e = int(threadIdx.x) + kTopThreads * q;
    if (e < K) {
      p.top[int64_t(ul) * p.n_top + e] = x[q];
      rp[x[q]] = e;
    }
  }
}

// Launched in clusters of 1 to 8 CTAs per unit; n_top at most kMaxE kTopThreads.
// (Where there are more units than SMs, two CTAs per SM cover each other's barriers: 32
// registers, which the sort of 4 or 8 keys per thread does not fit.  512 units of
// 16K keys, n_top = 64: 160 us -> 136.)
template <int kMaxE>
__global__ void __launch_bounds__(kTopThreads, kMaxE <= 2 ? 2 : 1) k_topk(TopArgs p) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) uint8_t smraw[];
  int n_sort = kTopThreads;                      // the power of two that holds n_top
  while (n_sort < p.n_top) n_sort *= 2;
  uint64_t* skey = reinterpret_cast<uint64_t*>(smraw);                   // [n_sort]
  int32_t* sidx = reinterpret_cast<int32_t*>(skey + n_sort);             // [n_sort]
  __shared__ int hist[kSelBins];
  __shared__ int warp_sums[32];
  __shared__ int64_t bcast[3];
  __shared__ int totals[2];                                               // keys above and at the threshold
  const int cs = int(cl.num_blocks()), rank = int(cl.block_rank());
  const int ul = int(blockIdx.x) / cs;
  const int64_t s = p.s;
  const int64_t n_ev = s > p.recent ? s - p.recent : 0;
  const double* sc = p.scores + int64_t(ul) * s;
  int32_t* rp = p.rank_pos + int64_t(ul) * s;
  int K = p.n_top;
  if (p.budgets) {
    const int64_t keep = (p.budgets[ul] < s ? int64_t(p.budgets[ul]) : s) - p.recent;
    K = keep < 0 ? 0 : int(keep);
    if (K > p.n_top) {
      if (threadIdx.x == 0 && rank == 0 && p.status) report_status(p.status, kStatusBadIndex);
      K = p.n_top;
    }
  }
  // protected window and default ranks
  for (int64_t i = s * rank / cs + threadIdx.x; i < s * (rank + 1) / cs; i += blockDim.x)
    rp[i] = (i < n_ev) ? INT_MAX : -1;
  if (K <= 0) return;                          // the whole cluster
  // this CTA's evictable positions; warp w takes a contiguous part of them
  const int64_t lo = n_ev * rank / cs, n = n_ev * (rank + 1) / cs - lo;
  const SelState st = cluster_select(cl, K, hist, warp_sums, bcast, [&](auto&& f) {
    for (int64_t i = threadIdx.x; i < n; i += kTopThreads) f(score_key(sc[lo + i]));
  });
  // order-preserving compaction: counts above and at the threshold per warp,
  // their places from the CTAs and warps before
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kTopThreads / 32;
  const int64_t w0 = lo + n * w / nw, w1 = lo + n * (w + 1) / nw;
  int n_gt = 0, n_eq = 0;
  for (int64_t i0 = w0; i0 < w1; i0 += 32) {
    const uint64_t key = i0 + lane < w1 ? score_key(sc[i0 + lane]) & st.mask : 0ull;
    n_gt += __popc(__ballot_sync(0xffffffffu, i0 + lane < w1 && key > st.prefix));
    n_eq += __popc(__ballot_sync(0xffffffffu, i0 + lane < w1 && key == st.prefix));
  }
  int tot_gt = 0, tot_eq = 0;
  int gt_before = block_exclusive_scan(lane == 0 ? n_gt : 0, warp_sums, &tot_gt);
  int eq_before = block_exclusive_scan(lane == 0 ? n_eq : 0, warp_sums, &tot_eq);
  gt_before = __shfl_sync(0xffffffffu, gt_before, 0);
  eq_before = __shfl_sync(0xffffffffu, eq_before, 0);
  if (threadIdx.x == 0) {
    totals[0] = tot_gt;
    totals[1] = tot_eq;
  }
  cl.sync();
  for (int r = 0; r < rank; ++r) {
    const int* o = cl.map_shared_rank(totals, r);
    gt_before += o[0];
    eq_before += o[1];
  }
  const int rem = int(st.rem);
  uint64_t* key0 = cl.map_shared_rank(skey, 0);
  int32_t* idx0 = cl.map_shared_rank(sidx, 0);
  for (int64_t i0 = w0; i0 < w1; i0 += 32) {
    const bool in = i0 + lane < w1;
    const uint64_t key = in ? score_key(sc[i0 + lane]) : 0ull;
    const bool gt = in && (key & st.mask) > st.prefix, eq = in && (key & st.mask) == st.prefix;
    const unsigned bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
    const unsigned below = (1u << lane) - 1u;
    const int eb = eq_before + __popc(be & below);             // equal keys before this one
    if (gt || (eq && eb < rem)) {
      const int out = gt_before + __popc(bg & below) + (eb < rem ? eb : rem);
      if (out < K) {
        key0[out] = key;
        idx0[out] = int32_t(i0 + lane);
      } else if (p.status) {
        report_status(p.status, kStatusBadIndex);
      }
    }
    gt_before += __popc(bg);
    eq_before += __popc(be);
  }
  cl.sync();                                   // the list is complete; nobody reads another CTA's memory after
  if (rank != 0) return;
  if (K <= kTopThreads) {
    topk_rank<1>(p, ul, K, skey, sidx);
  } else if (kMaxE == 2 || K <= 2 * kTopThreads) {
    topk_rank<2>(p, ul, K, skey, sidx);
  } else {
    if constexpr (kMaxE > 2) {
      if (K <= 4 * kTopThreads) topk_rank<4>(p, ul, K, skey, sidx);
      else topk_rank<8>(p, ul, K, skey, sidx);
    }
  }
}

// ---------------------------------------------------------------------------
// AdaKV budgets across the KV heads of one (layer, batch element) (App. B,
// "AdaKV": token scores as importance, safeguard coefficient).  Every head
// keeps |P| + f slots (its window and its f best-ranked tokens, which a
// ranking of the top f has marked in rank_pos); the n_free other slots go to
// the highest-scored remaining evictable tokens of all heads, ordered by
// (score desc, head asc, position asc).  One cluster per batch element: a radix
// select of the n_free-th largest key over the heads' remaining tokens, then
// per-head counts above and at the threshold.  (One CTA and eight 8-bit digits
// took 1043 us for 8 heads of 32K tokens, this with one load at a time 98, now 70.)
// ---------------------------------------------------------------------------

struct AdaArgs {
  const double* scores;      // [UL, s]
  const int32_t* rank_pos;   // [UL, s]: rank < f marks a head's safeguard tokens
  int64_t s;
  int32_t recent;            // |P| (clamped to s)
  int32_t n_heads;           // H_kv; unit ul = batch * H_kv + h
  int32_t f;                 // safeguard tokens per head
  int32_t base;              // |P| + f
  int64_t n_free;            // H_kv * (b - |P| - f)
  int32_t* budgets;          // [UL] out
  int32_t* counts;           // [UL, 2] scratch: tokens above and at the threshold
};

// Launched in clusters of 1 to 8 CTAs per batch element.
__global__ void __launch_bounds__(kTopThreads, 1) k_adakv(AdaArgs p) {
  cg::cluster_group cl = cg::this_cluster();
  __shared__ int hist[kSelBins];
  __shared__ int warp_sums[32];
  __shared__ int64_t bcast[3];
  const int cs = int(cl.num_blocks()), rank = int(cl.block_rank());
  const int grp = int(blockIdx.x) / cs, H = p.n_heads;
  const int64_t s = p.s, n_ev = s > p.recent ? s - p.recent : 0;
  const int ul0 = grp * H;
  if (p.n_free <= 0) {                          // the whole cluster
    for (int h = rank * kTopThreads + threadIdx.x; h < H; h += cs * kTopThreads) p.budgets[ul0 + h] = p.base;
    return;
  }
  for (int h = rank * kTopThreads + threadIdx.x; h < 2 * H; h += cs * kTopThreads) p.counts[2 * ul0 + h] = 0;
  // f(head, key) for the remaining tokens of this CTA's positions of every head
  const int64_t lo = n_ev * rank / cs, hi = n_ev * (rank + 1) / cs;
  // (eight loads in flight; not the head's safeguard tokens)
  auto each = [&](int h, auto&& f) {
    const double* sc = p.scores + int64_t(ul0 + h) * s;
    const int32_t* rp = p.rank_pos + int64_t(ul0 + h) * s;
    for (int64_t i = lo + threadIdx.x; i < hi; i += 8 * kTopThreads) {
      double v[8];
      bool take[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t x = i + j * kTopThreads;
        v[j] = x < hi ? __ldg(sc + x) : 0.0;
        take[j] = x < hi && __ldg(rp + x) >= p.f;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (take[j]) f(score_key(v[j]));
    }
  };
  const SelState st = cluster_select(cl, p.n_free, hist, warp_sums, bcast, [&](auto&& f) {
    for (int h = 0; h < H; ++h) each(h, f);
  });
  for (int h = 0; h < H; ++h) {
    int gt = 0, eq = 0;
    each(h, [&](uint64_t key) {
      gt += (key & st.mask) > st.prefix;
      eq += (key & st.mask) == st.prefix;
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      gt += __shfl_xor_sync(0xffffffffu, gt, o);
      eq += __shfl_xor_sync(0xffffffffu, eq, o);
    }
    if ((threadIdx.x & 31) == 0) {
      if (gt) atomicAdd(&p.counts[2 * (ul0 + h)], gt);
      if (eq) atomicAdd(&p.counts[2 * (ul0 + h) + 1], eq);
    }
  }
  __threadfence();
  cl.sync();
  if (rank != 0 || threadIdx.x != 0) return;
  // st.rem keys at the threshold are taken: lower heads first
  int64_t eq_before = 0;
  for (int h = 0; h < H; ++h) {
    const int gt = __ldcg(&p.counts[2 * (ul0 + h)]), eq = __ldcg(&p.counts[2 * (ul0 + h) + 1]);
    int64_t take_eq = st.rem - eq_before;
    take_eq = take_eq < 0 ? 0 : (take_eq > eq ? eq : take_eq);
    p.budgets[ul0 + h] = p.base + gt + int32_t(take_eq);
    eq_before += eq;
  }
}


// ---------------------------------------------------------------------------
// Residual entries by Lloyd's algorithm (Sec. 5.3, Eqs. residual_partition,
// summary; App. B: 4 iterations, initial centres = the highest-scored evicted
// keys).  One "run" builds r_unit[ul] entries for every unit of the layer.
// E = S \ M_r = { p < s - |P| : rank_pos[p] >= m - |P| },  m = b - r.
// Deterministic: assignments by (distance, centre index); exact integer member
// sums (fp64 in token order where a value has no fixed-point form); no float
// atomics.
// ---------------------------------------------------------------------------

constexpr int kMaxR = 8192;

// A launch works on n_units "runs of a unit": run unit u is unit u % UL of the
// layer, with candidate u / UL of the launch's.
struct LloydArgs {
  const __nv_bfloat16* K;      // layer keys [UL, s, d]
  const __nv_bfloat16* V;      // layer values
  int64_t s;
  int32_t UL;                  // (batch, KV head) units of the layer
  int32_t n_units;             // run units of this launch (U below)
  int32_t recent;              // |P| (already clamped to s)
  int32_t n_top;
  int32_t budget;
  int32_t ntiles;
  int32_t rmax;                // stride of the per-centre arrays, a multiple of 16
  const int32_t* top;          // [UL, n_top]
  const int32_t* rank_pos;     // [UL, s]
  const int32_t* budgets;      // [UL] per-unit budgets, or NULL (budget)
  const int32_t* r_unit;       // [U]
  float* cnorm;                // [U, rmax]     ||c||^2 of the fp32 copy; +inf from r to the
                               // next multiple of 16
  double* centers64;           // [U, rmax, d]  the centres (fp64 means)
  float* centers32;            // [U, rmax, d]  their fp32 copy
  __nv_bfloat16* cplanes;      // [U, 2 planes, 2 halves, rmax, 64] the fp32 centres split into two
                               // bf16 planes, laid out as the tensor cores read them (split_planes)
  float* knorm;                // [UL, s] an upper bound of every key's norm (the assignment's bound)
  int2* cand;                  // [U, s] candidates so far (units with more than one segment)
  int4* amb;                   // [U * ntiles * 128] tokens the assignment leaves to k_lloyd_resolve
  int* amb_count;              // their number, per assignment CTA
  int32_t* assign;             // [U, s] centre index, -1 outside E
  const int32_t* assign_prev;  // the iteration before, or NULL in the first (no token has a centre)
  int32_t* mcount;             // [U, 2, rmax] tokens that joined and that left a centre; zero before
                               // an assignment
  int32_t* cursor;             // [U, 2, rmax] of these, placed so far; zero before an assignment
  int32_t* ccount;             // [U, rmax] members per centre before this iteration
  int32_t* lbase;              // [U, 2, rmax] first list slot per group
  int32_t* lsize;              // [U] slots of the list
  int32_t* list;               // [U, 2 s] token positions: those that joined, grouped by centre, then
                               // those that left, grouped by centre (or every member, by centre)
  long long* msum;             // [U, rmax, 2, d] fixed-point member sums (K, V), dim 4 l + q at
                               // 32 q + l; zero between runs
  long long* tsum;             // [U, rmax, 2, d] what the fixed-point sums dropped, unit 2^-kTailBits
  uint32_t* mflag;             // [U, rmax] kSumTails: tsum holds a part of the sum; kSumFp64: a
                               // member value is outside both
  __nv_bfloat16* kbar;         // [UL, ent_stride, d] entries, candidate c's at run_off[c]
  __nv_bfloat16* vbar;
  int32_t* ecount;             // [UL, ent_stride]
  int64_t ent_stride;
  const int32_t* run_off;      // [candidates of the launch]
  uint32_t* status;
  int32_t test_fault;          // test hook: CTA 0's first column wait gives up
};

// The two bf16 planes of dims 4 lane .. 4 lane + 3 of centre j: c = c1 + c2 + e,
// |e| <= 2^-16 |c| (the remainder c - c1 is exact in fp32; each plane keeps 8
// significant bits).  A plane's 64-dim half is [rmax rows][128 bytes] with the
// 16-byte chunks of a row XOR-swizzled by the row, so that a bulk copy of rows
// is the tensor cores' K-major operand.
__device__ __forceinline__ void split_planes(const LloydArgs& p, int u, int j, int lane, const float (&c)[4]) {
  __nv_bfloat16 c1[4], c2[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c1[q] = __float2bfloat16_rn(c[q]);
    c2[q] = __float2bfloat16_rn(c[q] - __bfloat162float(c1[q]));
  }
  const int half = lane >> 4, ch = (lane & 15) >> 1;
  uint8_t* b = reinterpret_cast<uint8_t*>(p.cplanes) + ((int64_t(u) * 4 + half) * p.rmax + j) * 128 +
               ((ch ^ (j & 7)) << 4) + 8 * (lane & 1);
  *reinterpret_cast<uint2*>(b) = *reinterpret_cast<const uint2*>(c1);
  *reinterpret_cast<uint2*>(b + int64_t(p.rmax) * 256) = *reinterpret_cast<const uint2*>(c2);
}

constexpr int kFinWarps = 8;
constexpr int kFinScan = 8, kFinRows = 4;   // where a centre is summed in fp64: loads of assignments and of rows in flight

// centre j = key of the (m - |P| + j)-th ranked token, a warp each; the rows up
// to the next multiple of 16 become centres no token is near
__global__ void __launch_bounds__(kFinWarps * 32) k_lloyd_init(LloydArgs p) {
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * kFinWarps + (threadIdx.x >> 5), u = blockIdx.y, ul = u % p.UL;
  const int r = p.r_unit[u];
  if (j >= ((r + 15) & ~15)) return;
  const int64_t uj = int64_t(u) * p.rmax + j;
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  float n = INFINITY;
  if (j < r) {
    const int32_t keep = int32_t(unit_budget(p.budgets, ul, p.budget)) - r - p.recent;
    const int32_t pos = p.top[int64_t(ul) * p.n_top + keep + j];
    const uint2 w = *reinterpret_cast<const uint2*>(p.K + (int64_t(ul) * p.s + pos) * kHeadDim + 4 * lane);
    const float2 a = bf16x2_to_float2(w.x), b = bf16x2_to_float2(w.y);
    c[0] = a.x;
    c[1] = a.y;
    c[2] = b.x;
    c[3] = b.y;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      p.centers64[uj * kHeadDim + 4 * lane + q] = double(c[q]);
      p.centers32[uj * kHeadDim + 4 * lane + q] = c[q];
    }
    n = fmaf(c[3], c[3], fmaf(c[2], c[2], fmaf(c[1], c[1], c[0] * c[0])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  }
  split_planes(p, u, j, lane, c);
  if (lane == 0) p.cnorm[uj] = n;
}

// Tokens into lists grouped by centre (in any order inside a group: the member
// sums are integers).  kMembers = false: the tokens whose centre changed in this
// iteration, once by the centre they joined and once by the one they left (in the
// first iteration every evicted token joins); kMembers = true: every member by
// its centre.  A CTA takes 1024 kTok tokens of a unit: it counts them per group
// in shared memory, takes each group's place in its list with one atomic, and
// writes the positions.  The groups start at the exclusive prefix of their
// sizes, which every CTA of the unit forms again.  Dynamic shared memory: 4 r
// ints.
// What bounds it: the barriers and the prefix of every CTA, so a CTA takes 4096
// tokens where that still leaves two CTAs per SM (64 units of 32K keys: 26 -> 21
// us; 32 units of 128K: 47 -> 34; 512 of 16K: 75 -> 53), else 1024.
constexpr int kScatterThreads = 1024;

template <bool kMembers, int kTok>
__global__ void __launch_bounds__(kScatterThreads) k_lloyd_scatter(LloydArgs p) {
  extern __shared__ int sc_raw[];
  __shared__ int warp_sums[32];
  const int u = blockIdx.y;
  const int r = p.r_unit[u];
  if (r == 0) return;
  const int ng = kMembers ? r : 2 * r;       // groups
  int* cnt = sc_raw;                         // the CTA's tokens per group
  int* at = sc_raw + ng;                     // where they go
  const int64_t c0 = int64_t(u) * p.rmax;
  // size of group g, and its place in the [2, rmax] arrays
  auto slot = [&](int g) { return 2 * c0 + (g < r ? g : p.rmax + g - r); };
  auto size = [&](int g) {
    if constexpr (!kMembers) return p.mcount[slot(g)];
    else
      return (p.assign_prev ? p.ccount[c0 + g] : 0) + p.mcount[2 * c0 + g] - p.mcount[2 * c0 + p.rmax + g];
  };
  const int64_t pos0 = int64_t(blockIdx.x) * kTok * kScatterThreads + threadIdx.x;
  int a[kTok], o[kTok];                      // the tokens' centres now and before
#pragma unroll
  for (int t = 0; t < kTok; ++t) {
    const int64_t pos = pos0 + t * kScatterThreads;
    a[t] = o[t] = -1;
    if (pos < p.s) {
      a[t] = p.assign[int64_t(u) * p.s + pos];
      if (!kMembers && p.assign_prev) o[t] = p.assign_prev[int64_t(u) * p.s + pos];
    }
  }
  for (int g = threadIdx.x; g < ng; g += kScatterThreads) cnt[g] = 0;
  const int per = (ng + kScatterThreads - 1) / kScatterThreads, g0 = threadIdx.x * per;
  int mine = 0;
  for (int g = g0; g < min(g0 + per, ng); ++g) mine += size(g);
  int total = 0;
  int base = block_exclusive_scan(mine, warp_sums, &total);
  if (blockIdx.x == 0 && threadIdx.x == 0) p.lsize[u] = total;
  for (int g = g0; g < min(g0 + per, ng); ++g) {
    at[g] = base;
    if (blockIdx.x == 0) p.lbase[slot(g)] = base;
    base += size(g);
  }
  int ra[kTok], ro[kTok];
#pragma unroll
  for (int t = 0; t < kTok; ++t) {
    if (a[t] >= r || o[t] >= r) {            // only after a failed assignment
      report_status(p.status, kStatusBadIndex);
      a[t] = o[t] = -1;
    }
    if (!kMembers && a[t] == o[t]) a[t] = o[t] = -1;   // not moved
    ra[t] = a[t] >= 0 ? atomicAdd(&cnt[a[t]], 1) : 0;
    ro[t] = o[t] >= 0 ? atomicAdd(&cnt[r + o[t]], 1) : 0;
  }
  __syncthreads();
  for (int g = threadIdx.x; g < ng; g += kScatterThreads)
    if (cnt[g] > 0) at[g] += atomicAdd(p.cursor + slot(g), cnt[g]);
  __syncthreads();
  auto put = [&](int off, int t) {
    if (off < 0 || off >= 2 * p.s) {         // counts inconsistent with the assignment: the same
      report_status(p.status, kStatusBadIndex);
      return;
    }
    p.list[2 * int64_t(u) * p.s + off] = int32_t(pos0 + t * kScatterThreads);
  };
#pragma unroll
  for (int t = 0; t < kTok; ++t) {
    if (a[t] >= 0) put(at[a[t]] + ra[t], t);
    if (o[t] >= 0) put(at[r + o[t]] + ro[t], t);
  }
}

// New centre = mean key of its members; on the last iteration also the mean
// value, and the stored bf16 entry (Eq. summary).  The member sums are exact
// integers, so they are free of summation order, and the conversion of the
// total to fp64 is the exact sum rounded once; mean = that sum / count.
//
// Two kernels.  k_lloyd_accum sweeps the member list (grouped by centre)
// token-parallel: each warp takes kAccRowsPerWarp consecutive member slots,
// gathers their rows, keeps running sums for the centre it is in, and adds
// them into msum[ul][j] with 64-bit integer atomics when the centre changes.
// Integer addition is associative, so the totals do not depend on the order
// the atomics land in.  k_lloyd_finish then forms the means, one warp per
// centre, and clears the sums for the next pass.
//
// The running sum of a value is a pair of floats, S from C1 = 1.5 * 2^14 and T
// from C2 = 1.5 * 2^-3, added to without error while T's grid holds the value:
//   S' = S + x, h = S' - S, l = x - h   (Dekker's Fast2Sum, exact: |x| <= |S|)
//   T' = T + l, g = T' - T, e = l - g   (e: what T's grid, 2^-26, drops)
// so the sum is S + T - C1 - C2 exactly iff every e is zero.  S has to stay in
// its binade [2^14, 2^15), which its exponent bits tell after every addition
// (64 values below 128 always do): then |x| < 2^13 <= S, S is a multiple of 2^-9,
// |l| <= 2^-10, and T stays within 64 * 2^-10 of C2 and is a multiple of 2^-26, so
// both convert to integers of unit 2^-32.  Six packed fp32x2 additions and three ORs take two values
// through it, where the integer form this replaces took 8 additions, 2 integer
// additions and a maximum per value.
// A value is dropped from when it is below 2^-19 in magnitude (about 15 in
// 10^7 of normally distributed values, so in a few of a unit's centres): the
// warp then adds the exact e as 64-bit integers of unit 2^-59, kept beside and
// flushed into tsum.  |e| is at most half of T's grid, 2^32 units, so the 2^30
// members that a centre can have sum to 2^62 at most.  Sums that leave the binade
// (64 rows that sum past 8192) or values with bits below 2^-59 flag the centre: it
// is summed in fp64 in member order (k_lloyd_finish: its members are found and read
// a few loads at a time).  C1 is the least that holds 64 values below 128 (8 units of
// 32K keys, r = 51, a mean of 70 in one channel: 1.1 ms of iterations, with C1 = 1.5 *
// 2^13 11.4; a mean of 300, summed in fp64, 4.9 against 5.2 a row at a time).
constexpr int kAccRowsPerWarp = 64;
constexpr int kAccRows = kAccRowsPerWarp * (kThreads / 32);   // member slots per CTA
constexpr float kSumC1 = 24576.0f;
constexpr float kSumC2 = 0x1.8p-3f;
static_assert(kAccRowsPerWarp <= 64, "T must stay within 2^-4 of C2");
constexpr int kTailBits = 59;                                 // unit of a dropped part: 2^-59
constexpr float kTailScale = 0x1p59f;
enum : uint32_t { kSumFp64 = 1u, kSumTails = 2u };            // mflag

struct PairSum {
  float2 s, t;
};

__device__ __forceinline__ PairSum pair_zero() {
  return PairSum{make_float2(kSumC1, kSumC1), make_float2(kSumC2, kSumC2)};
}

// two values into their sums; returns what was dropped
__device__ __forceinline__ float2 pair_add(float2 x, PairSum& a) {
  const float2 s = fadd2(a.s, x), h = fsub2(s, a.s), l = fsub2(x, h);
  const float2 t = fadd2(a.t, l), g = fsub2(t, a.t);
  a.s = s;
  a.t = t;
  return fsub2(l, g);
}

// The fixed-point total of one sum, unit 2^-32 (exact).
__device__ __forceinline__ long long sum_total(float s, float t) {
  const long long c1 = 24576ll << 32, c2 = 3ll << 28;
  return (__float2ll_rz(s * 0x1p32f) - c1) + (__float2ll_rz(t * 0x1p32f) - c2);
}

// A dropped e as an integer of unit 2^-kTailBits; exact unless it has bits below.
__device__ __forceinline__ long long tail_units(float e, bool& ok) {
  const float x = e * kTailScale;
  const long long v = __float2ll_rz(x);
  ok &= fabsf(x) < 0x1p62f && __ll2float_rz(v) == x;
  return v;
}

// The lane's sums of four consecutive bf16 dims (two words, low half first).
struct RowSum {
  PairSum a, b;
  long long tail[4];             // the dropped parts, unit 2^-kTailBits
  uint32_t left;                 // OR of bits(S) ^ bits(C1)
  bool dropped, bad;             // some lane's e was not zero; an e has bits below its unit

  __device__ __forceinline__ void reset() {
    a = b = pair_zero();
    tail[0] = tail[1] = tail[2] = tail[3] = 0;
    left = 0u;
    dropped = bad = false;
  }
  // N rows, 32 words apart; every lane of the warp adds its part of them.
  // One vote covers the N rows: where something was dropped they are taken
  // once more for the exact e.
  template <int N>
  __device__ __forceinline__ void add(const uint2* w) {
    const PairSum a0 = a, b0 = b;
    const uint32_t c1 = __float_as_uint(kSumC1);
    uint32_t any = 0u;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const uint2 v = w[32 * q];
      const float2 e = pair_add(bf16x2_to_float2(v.x), a), f = pair_add(bf16x2_to_float2(v.y), b);
      left |= (__float_as_uint(a.s.x) ^ c1) | (__float_as_uint(a.s.y) ^ c1);
      left |= (__float_as_uint(b.s.x) ^ c1) | (__float_as_uint(b.s.y) ^ c1);
      any |= __float_as_uint(e.x) | __float_as_uint(e.y);
      any |= __float_as_uint(f.x) | __float_as_uint(f.y);
    }
    if (__any_sync(0xffffffffu, any != 0u)) {
      dropped = true;
      bool ok = true;
      PairSum ta = a0, tb = b0;
#pragma unroll 1
      for (int q = 0; q < N; ++q) {
        const uint2 v = w[32 * q];
        const float2 e = pair_add(bf16x2_to_float2(v.x), ta), f = pair_add(bf16x2_to_float2(v.y), tb);
        tail[0] += tail_units(e.x, ok);
        tail[1] += tail_units(e.y, ok);
        tail[2] += tail_units(f.x, ok);
        tail[3] += tail_units(f.y, ok);
      }
      bad |= !ok;
    }
  }
  // whether a sum left its binade (its sign or exponent bits changed)
  __device__ __forceinline__ bool out_of_range() const { return (left & 0xff800000u) != 0u; }
};

// values = false: the key sums, updated by the tokens that joined a centre and
// those that left one (the list of k_lloyd_scatter<false>; integer sums, so the
// update is exact; in the first iteration every member joins).  values = true: the
// value sums of every member (the last iteration, k_lloyd_scatter<true>).  wide: the
// rows lie on a 16-byte boundary.  A value
// without a fixed-point form that joins raises the centre's flag, which stays for
// the run (a flagged centre is summed again in fp64 from its members).
// What bounds it: instruction issue (about 40 warp instructions per 256-byte row,
// 2.7 issued per cycle) and DRAM, at 58 % of its rate.  A warp's rows arrive by
// cp.async in a ring of kAccDepth batches of 8 (2 KB each), so that 8 KB per
// warp and about 190 KB per SM are in flight whatever its registers; rows of
// one centre are added four at a time without a look at the centre's end or at
// what was dropped in between.  A full pass over 64 units of 32K keys (2.03 M
// rows of 256 B, r = 51..204) takes 118 us; the integer form, whose loads went
// through registers, took 176.
constexpr int kAccDepth = 4;
constexpr size_t kAccSmem = size_t(kThreads / 32) * kAccDepth * 8 * kAsgRowBytes;

template <bool values, bool wide>
__global__ void __launch_bounds__(kThreads, 3) k_lloyd_accum(LloydArgs p) {
  extern __shared__ __align__(128) uint8_t acc_raw[];
  __shared__ int rows_s[kThreads / 32][kAccRowsPerWarp];   // positions of the rows to add
  const int u = blockIdx.y;
  const int r = p.r_unit[u];
  if (r <= 0) return;
  const int64_t c0 = int64_t(u) * p.rmax;
  // groups of the list: joined (or every member) by centre, then left by centre
  const int ng = values || !p.assign_prev ? r : 2 * r;
  auto slot = [&](int g) { return 2 * c0 + (g < r ? g : p.rmax + g - r); };
  // (the clamps below only act after a failed assignment, whose status is raised)
  const int n_list = int(min(int64_t(p.lsize[u]), 2 * p.s));
  auto start = [&](int g) { return p.lbase[slot(g)]; };
  auto end = [&](int g) { return g + 1 < ng ? start(g + 1) : n_list; };
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const __nv_bfloat16* X = (values ? p.V : p.K) + int64_t(u % p.UL) * p.s * kHeadDim;
  int* rows = rows_s[w];
  for (int lo = blockIdx.x * kAccRows + w * kAccRowsPerWarp; lo < n_list; lo += gridDim.x * kAccRows) {
    const int n = min(n_list - lo, kAccRowsPerWarp);
    // (a position outside the unit only follows a failed assignment: row 0 is
    // read instead of leaving the array)
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kAccRowsPerWarp / 32; ++k) {
      const int x = 32 * k + lane;
      const int pos = x < n ? p.list[2 * int64_t(u) * p.s + lo + x] : 0;
      rows[x] = uint32_t(pos) < uint32_t(p.s) ? pos : 0;
    }
    __syncwarp();
    const uint32_t ring = smem_u32(acc_raw) + uint32_t(w * kAccDepth * 8 * kAsgRowBytes);
    const uint2* ringp = reinterpret_cast<const uint2*>(acc_raw + w * kAccDepth * 8 * kAsgRowBytes) + lane;
    // rows 8b .. 8b + 7 into stage b % kAccDepth: half a warp per row (rows on
    // an 8-byte boundary only, which keys and values may lie on: two copies a lane)
    auto issue = [&](int b) {
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        const int x = 8 * b + q + (lane >> 4);
        if (x < n) {
          const uint32_t dst = ring + uint32_t(((b % kAccDepth) * 8 + q + (lane >> 4)) * kAsgRowBytes + (lane & 15) * 16);
          const __nv_bfloat16* src = X + int64_t(rows[x]) * kHeadDim + 8 * (lane & 15);
          if constexpr (wide) {
            cp_async16(dst, src, 16u);
          } else {
            cp_async8(dst, src);
            cp_async8(dst + 8, src + 4);
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int b = 0; b < kAccDepth; ++b) issue(b);
    // the group holding slot lo: the last one that starts at or before it (it is
    // never empty: an empty group starts with the next one)
    int j = 0;
    for (int step = 1 << (31 - __clz(max(ng - 1, 1))); step > 0; step >>= 1)
      if (j + step < ng && start(j + step) <= lo) j += step;
    int bnd = end(j) - lo;          // the row after the group's last
    const int64_t m0 = c0 * 2 * kHeadDim + (values ? kHeadDim : 0) + lane;
    unsigned long long* ms = reinterpret_cast<unsigned long long*>(p.msum) + m0;
    unsigned long long* ts = reinterpret_cast<unsigned long long*>(p.tsum) + m0;
    RowSum sum;
    sum.reset();
    // the lane's sums into group jj's centre (dim 4 lane + q at 32 q + lane, so
    // that a warp's additions meet whole sectors)
    auto flush = [&](int jj) {
      const bool left = jj >= r;
      const int c = left ? jj - r : jj;
      unsigned long long* m = ms + int64_t(c) * 2 * kHeadDim;
      const long long v[4] = {sum_total(sum.a.s.x, sum.a.t.x), sum_total(sum.a.s.y, sum.a.t.y),
                              sum_total(sum.b.s.x, sum.b.t.x), sum_total(sum.b.s.y, sum.b.t.y)};
#pragma unroll
      for (int q = 0; q < 4; ++q) atomicAdd(m + 32 * q, static_cast<unsigned long long>(left ? -v[q] : v[q]));
      const bool bad = __any_sync(0xffffffffu, sum.bad || sum.out_of_range());
      if (sum.dropped) {
        unsigned long long* t = ts + int64_t(c) * 2 * kHeadDim;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (sum.tail[q] != 0)
            atomicAdd(t + 32 * q, static_cast<unsigned long long>(left ? -sum.tail[q] : sum.tail[q]));
      }
      if ((sum.dropped || bad) && lane == 0)
        atomicOr(p.mflag + c0 + c, (sum.dropped ? kSumTails : 0u) | (bad ? kSumFp64 : 0u));
      sum.reset();
    };
    for (int b = 0; 8 * b < n; ++b) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kAccDepth - 1) : "memory");
      __syncwarp();
      const uint2* st = ringp + (b % kAccDepth) * 8 * 32 - 8 * b * 32;      // row x at st + 32 x
      const int xe = min(n, 8 * b + 8);
      for (int x = 8 * b; x < xe;) {
        if (x >= bnd && j < ng - 1) {               // warp-uniform: row x is of a later group
          if (x > 0) flush(j);
          do {
            ++j;
            bnd = end(j) - lo;
          } while (x >= bnd && j < ng - 1);
        }
        const int xs = j < ng - 1 ? min(xe, bnd) : xe;
        for (; x + 4 <= xs; x += 4) sum.add<4>(st + 32 * x);
        for (; x < xs; ++x) sum.add<1>(st + 32 * x);
      }
      __syncwarp();
      issue(b + kAccDepth);
    }
    flush(j);
  }
}

// One warp per centre, lane l on dims 4l..4l+3 (coalesced sums, centres and
// entries); ||c||^2 of the fp32 centre by a butterfly (the certification
// bounds its rounding for any summation order).
__global__ void __launch_bounds__(kFinWarps * 32) k_lloyd_finish(LloydArgs p, int final_pass) {
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * kFinWarps + (threadIdx.x >> 5), u = blockIdx.y, ul = u % p.UL;
  const int r = p.r_unit[u];
  // members of the block's centres and their rounded reciprocals: one fp64
  // division for all of them
  __shared__ int cnt_s[kFinWarps];
  __shared__ int mem_s[kFinWarps][32 * kFinScan + kFinRows];
  __shared__ double rcp_s[kFinWarps];
  if (threadIdx.x < kFinWarps) {
    const int jj = blockIdx.x * kFinWarps + threadIdx.x;
    int n = 0;
    if (jj < r) {
      const int32_t* mc = p.mcount + 2 * int64_t(u) * p.rmax + jj;
      n = (p.assign_prev ? p.ccount[int64_t(u) * p.rmax + jj] : 0) + mc[0] - mc[p.rmax];
    }
    cnt_s[threadIdx.x] = n;
    rcp_s[threadIdx.x] = n > 0 ? (1.0 / double(n)) * 0x1p-32 : 0.0;
  }
  __syncthreads();
  if (j >= r) return;
  const int64_t uj = int64_t(u) * p.rmax + j;
  const int cnt = cnt_s[threadIdx.x >> 5];
  const uint32_t flag = p.mflag[uj];
  const bool exact = flag == 0u;
  // dim 4 lane + q of the key sums at 32 q, of the value sums at kHeadDim + 32 q
  long long* ms = p.msum + uj * 2 * kHeadDim + lane;
  long long* ts = p.tsum + uj * 2 * kHeadDim + lane;
  // mean = RN(sum / cnt) with sum = RN(S * 2^-32) for the integer sum S: by
  // Markstein's correction with the rounded reciprocal y = RN(1 / (cnt 2^32)),
  // q0 = RN(S y), r = S - q0 cnt 2^32 (exact in one fma), q = RN(q0 + r y) is
  // the correctly rounded quotient -- two fp64 fmas and a product per
  // dimension instead of a division (fp64 is scarce on this part)
  double tk[4], tv[4], mk[4], mv[4];
  const double cd = double(cnt);
  if (exact) {
    const double y = rcp_s[threadIdx.x >> 5];
    const double bd = cd * 0x1p32;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double sk = double(ms[32 * q]);
      const double qk = sk * y;
      mk[q] = fma(fma(-qk, bd, sk), y, qk);
      mv[q] = 0.0;
      if (final_pass) {
        const double sv = double(ms[kHeadDim + 32 * q]);
        const double qv = sv * y;
        mv[q] = fma(fma(-qv, bd, sv), y, qv);
      }
    }
  } else if ((flag & kSumFp64) == 0u) {
    // some values have bits below T's grid: sum = RN(S * 2^-32 + tails * 2^-kTailBits),
    // the quotient formed as above (divisions and 128-bit sums for one centre in ten
    // cost the kernel 1.3 to 2.4 us of its 12 to 31)
    const double y = rcp_s[threadIdx.x >> 5] * 0x1p32;
    auto mean = [&](long long hi, long long lo) {
      double x;
      if (llabs(hi) < (1ll << 53) && llabs(lo) < (1ll << 53)) {
        x = fma(double(lo), 1.0 / double(1ll << kTailBits), double(hi) * 0x1p-32);   // both exact: rounded once
      } else {
        const __int128 v = (__int128(hi) << (kTailBits - 32)) + lo;
        const double a = v == 0 ? 0.0 : round_u128(u128(v < 0 ? -v : v), -kTailBits, false);
        x = v < 0 ? -a : a;
      }
      const double q0 = x * y;
      return fma(fma(-q0, cd, x), y, q0);
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      mk[q] = mean(ms[32 * q], ts[32 * q]);
      mv[q] = final_pass ? mean(ms[kHeadDim + 32 * q], ts[kHeadDim + 32 * q]) : 0.0;
    }
  } else {
    // fp64 sums over the unit's tokens in order
#pragma unroll
    for (int q = 0; q < 4; ++q) tk[q] = tv[q] = 0.0;
    const int32_t* as = p.assign + int64_t(u) * p.s;
    const __nv_bfloat16* Kd = p.K + int64_t(ul) * p.s * kHeadDim + 4 * lane;
    const __nv_bfloat16* Vd = p.V + int64_t(ul) * p.s * kHeadDim + 4 * lane;
    int* mem = mem_s[threadIdx.x >> 5];           // members found and not yet added
    int found = 0;
    // rows mem[i .. i + kFinRows - 1] of X (below n) into t
    auto add_rows = [&](const __nv_bfloat16* X, int i, int n, double (&t)[4]) {
      uint2 w[kFinRows];
#pragma unroll
      for (int q = 0; q < kFinRows; ++q)
        if (i + q < n) w[q] = __ldg(reinterpret_cast<const uint2*>(X + int64_t(mem[i + q]) * kHeadDim));
#pragma unroll
      for (int q = 0; q < kFinRows; ++q)
        if (i + q < n) {
          const float2 a = bf16x2_to_float2(w[q].x), b = bf16x2_to_float2(w[q].y);
          t[0] += double(a.x);
          t[1] += double(a.y);
          t[2] += double(b.x);
          t[3] += double(b.y);
        }
    };
    for (int64_t t0 = 0; t0 < p.s; t0 += 32 * kFinScan) {
      int a[kFinScan];
#pragma unroll
      for (int k = 0; k < kFinScan; ++k) {
        const int64_t pos = t0 + 32 * k + lane;
        a[k] = pos < p.s ? __ldg(as + pos) : -1;
      }
#pragma unroll
      for (int k = 0; k < kFinScan; ++k) {
        const unsigned take = __ballot_sync(0xffffffffu, a[k] == j);
        if (a[k] == j) mem[found + __popc(take & ((1u << lane) - 1u))] = int(t0) + 32 * k + lane;
        found += __popc(take);
      }
      __syncwarp();
      const int n = t0 + 32 * kFinScan < p.s ? found & ~(kFinRows - 1) : found;
      for (int i = 0; i < n; i += kFinRows) {
        add_rows(Kd, i, n, tk);
        if (final_pass) add_rows(Vd, i, n, tv);
      }
      // (fewer than kFinRows left)
      const int left = lane < found - n ? mem[n + lane] : 0;
      __syncwarp();
      if (lane < found - n) mem[lane] = left;
      found -= n;
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      mk[q] = tk[q] / cd;
      mv[q] = final_pass ? tv[q] / cd : 0.0;
    }
  }
  if (final_pass) {                   // the next run starts from zero
#pragma unroll
    for (int q = 0; q < 4; ++q) ms[32 * q] = ms[kHeadDim + 32 * q] = 0;
    if (!exact) {
#pragma unroll
      for (int q = 0; q < 4; ++q) ts[32 * q] = ts[kHeadDim + 32 * q] = 0;
    }
  }
  double* c64 = p.centers64 + uj * kHeadDim + 4 * lane;
  float* c32 = p.centers32 + uj * kHeadDim + 4 * lane;
  float cf[4];
  if (cnt > 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cf[q] = float(mk[q]);
      c64[q] = mk[q];
      c32[q] = cf[q];
    }
    split_planes(p, u, j, lane, cf);
  } else {                            // an empty centre keeps its place
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      mk[q] = c64[q];
      cf[q] = c32[q];
    }
  }
  float n = fmaf(cf[3], cf[3], fmaf(cf[2], cf[2], fmaf(cf[1], cf[1], cf[0] * cf[0])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if (final_pass) {
    const int64_t e = int64_t(ul) * p.ent_stride + p.run_off[u / p.UL] + j;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      p.kbar[e * kHeadDim + 4 * lane + q] = __double2bfloat16(mk[q]);
      p.vbar[e * kHeadDim + 4 * lane + q] = __double2bfloat16(cnt > 0 ? mv[q] : 0.0);
    }
    if (lane == 0) p.ecount[e] = cnt;
  }
  __syncwarp();                       // every lane has read mflag
  if (lane == 0) {
    p.cnorm[uj] = n;
    p.ccount[uj] = cnt;
    if (final_pass) p.mflag[uj] = 0u;
  }
}

// ---------------------------------------------------------------------------
// Validation proxy (Sec. 5.5.1, Eqs. valloss, valproxy; Alg. 1)
// ---------------------------------------------------------------------------

constexpr int kValRec = kHeadDim + 4;        // m, l, 2 pad, acc[d]: acc 16-byte aligned
constexpr int kValRows = 128;                // query rows per CTA, at most

// Attention of the validation queries over many tokens on the tensor cores
// (mma.sync m16n8k16, as the scores), shared by the targets (k_val_full) and the
// candidates' losses (k_val_loss).  A CTA of 8 warps walks tiles of 128 key and
// value rows (bf16, 256-byte rows XOR-swizzled for ldmatrix), two in flight by
// cp.async.  The warps split the query rows in groups of 16 and, where there are
// fewer than 8 groups, each tile's tokens between `splits` warps of a group.  A
// warp takes 32 tokens at a time: logits (exact bf16 products, fp32 sums), an
// online softmax in registers, and P V with the fp32 weights split into three
// bf16 planes (p = p1 + p2 + p3 exactly), so no weight loses a bit.  The sums of
// 32 tokens are formed apart and added to the running ones in fp32: longer chains
// of tensor-core additions, which do not round to nearest, had twice the error of
// the fp32 FMAs this replaces against 64 bits; so formed it is the same (mean error
// of L_0 over 6 shapes 3.8e-7 of it, before and now).
//
// What bounds it: the legacy tensor-core rate (four times the products of one
// bf16 plane) and the softmax's issue between the MMAs.  P V used to take fp32
// FMAs from shared memory, with half of the warps idle during the logits:
// targets of 64 units x 32 rows x 32K tokens 645 -> 320 us, of 32 units x 128 rows
// x 128K tokens 4822 -> 1769 us; five columns of losses (b = 1024, batch 8) 508 ->
// 142 us a layer, in one launch.
struct ValState {
  float O[16][4];                // numerators of rows g, g + 8 at dims 8 nt + 2 t4 (+1)
  float m[2], l[2];              // reference maxima, this lane's share of the sums

  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) O[nt][0] = O[nt][1] = O[nt][2] = O[nt][3] = 0.f;
    m[0] = m[1] = -INFINITY;
    l[0] = l[1] = 0.f;
  }
};

// D = A * B, m16n8k16, bf16 inputs, fp32 result
__device__ __forceinline__ void mma16816_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// How a CTA's warps share its rows and a tile's tokens.
struct ValShape {
  int groups;                    // groups of 16 rows: 1, 2, 4 or 8
  int splits;                    // warps per group: min(4, 8 / groups)
};

__host__ __device__ inline ValShape val_shape(int n_rows) {
  const int g = (n_rows + 15) / 16;
  ValShape v;
  v.groups = g <= 1 ? 1 : g <= 2 ? 2 : g <= 4 ? 4 : 8;
  v.splits = v.groups >= 2 ? 8 / v.groups : 4;
  return v;
}

// A fragments (m16n8k16) of 16 query rows: row g and g + 8 of lane g = lane / 4
// from rowptr(i) (nullptr: a zero row), unscaled bf16
template <typename RowPtr>
__device__ __forceinline__ void val_afrag(RowPtr rowptr, int lane, uint32_t (&A)[8][4]) {
  const int g = lane >> 2, t4 = lane & 3;
  const uint32_t* q0 = reinterpret_cast<const uint32_t*>(rowptr(g));
  const uint32_t* q1 = reinterpret_cast<const uint32_t*>(rowptr(g + 8));
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    A[ks][0] = q0 ? __ldg(q0 + 8 * ks + t4) : 0u;
    A[ks][1] = q1 ? __ldg(q1 + 8 * ks + t4) : 0u;
    A[ks][2] = q0 ? __ldg(q0 + 8 * ks + 4 + t4) : 0u;
    A[ks][3] = q1 ? __ldg(q1 + 8 * ks + 4 + t4) : 0u;
  }
}

// 128 rows of 256 bytes into a swizzled bf16 tile by cp.async, one 16-byte chunk
// per copy; rowptr(i) = nullptr: zeros (the copy then reads nothing from `any`, a
// valid global address)
template <typename RowPtr>
__device__ __forceinline__ void val_stage_rows(uint32_t dst, RowPtr rowptr, const __nv_bfloat16* any) {
  for (int idx = threadIdx.x; idx < kTile * 16; idx += blockDim.x) {
    const int row = idx >> 4, ch = idx & 15;
    const __nv_bfloat16* src = rowptr(row);
    cp_async16(dst + asg_swz(row, ch), src ? src + 8 * ch : any, src ? 16u : 0u);
  }
}

// Tokens tk .. tk + 31 of the staged tile (keys at ks_s, values at vs_s) into
// st; bias (log2 units, -inf: no token) per token of the tile, or NULL.
__device__ __forceinline__ void val_block(ValState& st, const uint32_t (&A)[8][4], uint32_t ks_s, uint32_t vs_s,
                                          int tk, const float* bias) {
  const int lane = threadIdx.x & 31, t4 = lane & 3, mi = lane >> 3;
  float S[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) S[nt][0] = S[nt][1] = S[nt][2] = S[nt][3] = 0.f;
#pragma unroll
  for (int np = 0; np < 2; ++np) {
    const int trow = tk + 16 * np + (mi >> 1) * 8 + (lane & 7);
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t b0, b1, b2, b3;
      ldsm_x4(ks_s + asg_swz(trow, 2 * ks + (mi & 1)), b0, b1, b2, b3);
      mma16816(S[2 * np], A[ks][0], A[ks][1], A[ks][2], A[ks][3], b0, b1);
      mma16816(S[2 * np + 1], A[ks][0], A[ks][1], A[ks][2], A[ks][3], b2, b3);
    }
  }
  const float scale = kLog2e * rsqrtf(float(kHeadDim));
  float mx[2] = {st.m[0], st.m[1]};
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
    float2 bs = make_float2(0.f, 0.f);
    if (bias) bs = *reinterpret_cast<const float2*>(bias + tk + 8 * nt + 2 * t4);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      S[nt][2 * a] = fmaf(S[nt][2 * a], scale, bs.x);
      S[nt][2 * a + 1] = fmaf(S[nt][2 * a + 1], scale, bs.y);
      mx[a] = fmaxf(mx[a], fmaxf(S[nt][2 * a], S[nt][2 * a + 1]));
    }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], 1));
    mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], 2));
  }
  if (__any_sync(0xffffffffu, mx[0] > st.m[0] || mx[1] > st.m[1])) {
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      // (no token so far and none here: mx = -inf, nothing to scale)
      const float sc = mx[a] == -INFINITY ? 1.0f : exp2f(st.m[a] - mx[a]);
      st.m[a] = mx[a];
      st.l[a] *= sc;
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) {
        st.O[nt][2 * a] *= sc;
        st.O[nt][2 * a + 1] *= sc;
      }
    }
  }
  float ls[4][2];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int a = 0; a < 2; ++a) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
        S[nt][2 * a + c] = st.m[a] == -INFINITY ? 0.f : exp2f(S[nt][2 * a + c] - st.m[a]);
      ls[nt][a] = S[nt][2 * a] + S[nt][2 * a + 1];
    }
#pragma unroll
  for (int a = 0; a < 2; ++a) st.l[a] += (ls[0][a] + ls[1][a]) + (ls[2][a] + ls[3][a]);
  // the weights' three planes: n-tiles 2j, 2j + 1 are the A fragment of tokens 16j ..
  uint32_t P[2][3][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      float x = S[2 * j + (f >> 1)][2 * (f & 1)], y = S[2 * j + (f >> 1)][2 * (f & 1) + 1];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        P[j][pl][f] = pack_bf16(x, y);
        const float2 h = unpack_bf16(P[j][pl][f]);
        x -= h.x;
        y -= h.y;
      }
    }
  const int vrow = tk + (mi & 1) * 8 + (lane & 7);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    uint32_t v[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
      ldsm_x4_t(vs_s + asg_swz(vrow + 16 * j, 2 * q + (mi >> 1)), v[j][0], v[j][1], v[j][2], v[j][3]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {                // the smallest products first
      float T[4];
      mma16816_zero(T, P[0][2], v[0][2 * h], v[0][2 * h + 1]);
      mma16816(T, P[1][2][0], P[1][2][1], P[1][2][2], P[1][2][3], v[1][2 * h], v[1][2 * h + 1]);
#pragma unroll
      for (int pl = 1; pl >= 0; --pl)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          mma16816(T, P[j][pl][0], P[j][pl][1], P[j][pl][2], P[j][pl][3], v[j][2 * h], v[j][2 * h + 1]);
#pragma unroll
      for (int e = 0; e < 4; ++e) st.O[2 * q + h][e] += T[e];
    }
  }
}

// The warp's part of a staged tile.
__device__ __forceinline__ void val_tile(ValState& st, const uint32_t (&A)[8][4], uint32_t ks_s, uint32_t vs_s,
                                         int split, int splits, const float* bias) {
  const int n = kTile / splits;                  // this warp's tokens
  for (int tk = split * n; tk < (split + 1) * n; tk += 32) val_block(st, A, ks_s, vs_s, tk, bias);
}

// The finished state as records (m, l, pad, pad, acc) of the warp's 16 rows;
// rec(row) is row's record.
template <typename Rec>
__device__ __forceinline__ void val_store(ValState& st, Rec rec) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    float l = st.l[a];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    float* r = rec(g + 8 * a);
    if (!r) continue;
    if (t4 == 0) *reinterpret_cast<float2*>(r) = make_float2(st.m[a], l);
#pragma unroll
    for (int nt = 0; nt < 16; ++nt)
      *reinterpret_cast<float2*>(r + 4 + 8 * nt + 2 * t4) = make_float2(st.O[nt][2 * a], st.O[nt][2 * a + 1]);
  }
}

// Dynamic shared memory: two stages of a key and a value tile, their biases, and
// (k_val_loss) the records of the main branch.
constexpr size_t kValStage = 2 * size_t(kTile) * kAsgRowBytes;
constexpr size_t kValOffBias = 2 * kValStage;
constexpr size_t kValOffRec = kValOffBias + 2 * kTile * 4;
constexpr size_t kValSmemFull = kValOffRec;
constexpr size_t kValSmemLoss = kValOffRec + size_t(kThreads / 32) * 16 * kValRec * 4;
static_assert(size_t(kThreads / 32) * 16 * kValRec * 4 <= kValOffBias, "the residual records reuse the stages");

struct ValArgs {
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  const __nv_bfloat16* Qobs;   // [UL*G, n_obs, d]
  int64_t s;
  int32_t G, n_obs, n_val, n_rows;     // n_rows = G * n_val, row = g * n_val + t
  int32_t chunk_tiles;         // tiles per CTA
  int32_t nchunks;
  int32_t nparts;              // partial records per row: chunks x the last row block's splits
  float* part;                 // [UL, n_rows, nparts, kValRec]  (m, l, pad, acc)
  float* oS;                   // [UL, n_rows, d]
};

// Query row `row` of unit ul: the last n_val observation rows of its heads.
template <typename Args>
__device__ __forceinline__ const __nv_bfloat16* val_row(const Args& p, int ul, int row) {
  const int g = row / p.n_val, t = row % p.n_val;
  return p.Qobs + ((int64_t(ul) * p.G + g) * p.n_obs + (p.n_obs - p.n_val) + t) * kHeadDim;
}

// o_S(q) over all s tokens for the validation queries (Eq. attn), per chunk
__global__ void __launch_bounds__(kThreads, 1) k_val_full(ValArgs p) {
  extern __shared__ __align__(1024) uint8_t vraw[];
  const uint32_t st_s = smem_u32(vraw);
  float* bias_s = reinterpret_cast<float*>(vraw + kValOffBias);
  const int chunk = blockIdx.x, rb = blockIdx.y * kValRows, ul = blockIdx.z;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const ValShape sh = val_shape(min(kValRows, p.n_rows - rb));
  const int grp = w / sh.splits, split = w % sh.splits;
  const bool active = grp < sh.groups;
  const int r16 = rb + 16 * grp;
  uint32_t A[8][4];
  val_afrag([&](int i) { return active && r16 + i < p.n_rows ? val_row(p, ul, r16 + i) : nullptr; }, lane, A);
  const __nv_bfloat16* Ku = p.K + int64_t(ul) * p.s * kHeadDim;
  const __nv_bfloat16* Vu = p.V + int64_t(ul) * p.s * kHeadDim;
  const int64_t tile0 = int64_t(chunk) * p.chunk_tiles;
  const int n = int(min(int64_t(p.chunk_tiles), (p.s + kTile - 1) / kTile - tile0));
  auto issue = [&](int t) {                      // tile t of the chunk into stage t & 1
    if (t < n) {
      const int64_t tok0 = (tile0 + t) * kTile;
      const uint32_t dst = st_s + uint32_t((t & 1) * kValStage);
      val_stage_rows(dst, [&](int i) { return tok0 + i < p.s ? Ku + (tok0 + i) * kHeadDim : nullptr; }, Ku);
      val_stage_rows(dst + kTile * kAsgRowBytes,
                     [&](int i) { return tok0 + i < p.s ? Vu + (tok0 + i) * kHeadDim : nullptr; }, Vu);
      if (tok0 + kTile > p.s && threadIdx.x < kTile)
        bias_s[(t & 1) * kTile + threadIdx.x] = tok0 + threadIdx.x < p.s ? 0.f : -INFINITY;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  ValState st;
  st.reset();
  issue(0);
  for (int t = 0; t < n; ++t) {
    issue(t + 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const uint32_t ks_s = st_s + uint32_t((t & 1) * kValStage);
    const bool ragged = (tile0 + t + 1) * kTile > p.s;
    if (active)
      val_tile(st, A, ks_s, ks_s + kTile * kAsgRowBytes, split, sh.splits,
               ragged ? bias_s + (t & 1) * kTile : nullptr);
    __syncthreads();
  }
  if (active)
    val_store(st, [&](int i) -> float* {
      const int row = r16 + i;
      return row < p.n_rows ? p.part + ((int64_t(ul) * p.n_rows + row) * p.nparts + chunk * sh.splits + split) * kValRec
                            : nullptr;
    });
}

__global__ void k_val_combine(ValArgs p) {
  const int row = blockIdx.x, ul = blockIdx.y, d = threadIdx.x;
  const float* base = p.part + (int64_t(ul) * p.n_rows + row) * p.nparts * kValRec;
  const int n = p.nchunks * val_shape(min(kValRows, p.n_rows - row / kValRows * kValRows)).splits;
  float m = -INFINITY, l = 0.f, a = 0.f;
#pragma unroll 4
  for (int c = 0; c < n; ++c) {
    const float* q = base + int64_t(c) * kValRec;
    const float cm = q[0], cl = q[1], ca = q[4 + d];
    if (cl <= 0.f) continue;
    const float mn = fmaxf(m, cm);
    const float s0 = exp2f(m - mn), s1 = exp2f(cm - mn);
    l = l * s0 + cl * s1;
    a = a * s0 + ca * s1;
    m = mn;
  }
  p.oS[(int64_t(ul) * p.n_rows + row) * kHeadDim + d] = a / l;
}

struct LossArgs {
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  const __nv_bfloat16* Qobs;
  int64_t s;
  int32_t UL;
  int32_t G, n_obs, n_val, n_rows;
  int32_t recent, n_top, budget;
  const int32_t* top;          // [UL, n_top]
  const int32_t* r_runs;       // [runs, UL]: r of every candidate; run 0: the pure main cache
  const __nv_bfloat16* kbar;   // [UL, ent_stride, d], run k's entries at run_off[k]
  const __nv_bfloat16* vbar;
  const int32_t* ecount;
  int64_t ent_stride;
  const int32_t* run_off;
  float beta;
  int32_t gate_mode;
  float tau, alpha, g_min, g_fixed;
  const float* oS;             // [UL, n_rows, d]
  double* rowerr;              // [runs, UL, n_rows]
  int32_t softmax_mode;        // decode rule of the losses (RESKV_SOFTMAX_*)
  const int32_t* budgets;      // [UL] per-unit budgets, or NULL (budget)
};

// ||o^(r)(q) - o_S(q)||^2 per validation query and candidate, with the decode
// rule of Sec. 5.4 and the gate.  A CTA takes up to 128 query rows of a unit and
// one candidate: it walks the candidate's main slots (the kept ranked tokens,
// then the recent window), then its residual entries (logit + beta ln c), each
// gathered into shared memory once for all rows; one softmax state per branch,
// the main one kept in shared memory while the residual one runs.
__global__ void __launch_bounds__(kThreads, 1) k_val_loss(LossArgs p) {
  extern __shared__ __align__(1024) uint8_t vraw[];
  const uint32_t st_s = smem_u32(vraw);
  float* bias_s = reinterpret_cast<float*>(vraw + kValOffBias);
  float* rec_m = reinterpret_cast<float*>(vraw + kValOffRec);     // [8 warps][16 rows][kValRec]
  float* rec_r = reinterpret_cast<float*>(vraw);                  // the same, over the stages
  const int rb = blockIdx.x * kValRows, ul = blockIdx.y, run = blockIdx.z;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = p.r_runs[int64_t(run) * p.UL + ul];
  if (run > 0 && r == 0) return;                 // the unit has no such candidate
  const int64_t bu = unit_budget(p.budgets, ul, p.budget);
  const int64_t m = r == 0 ? (bu < p.s ? bu : p.s) : bu - r;
  const int64_t keep = m - p.recent;
  const ValShape sh = val_shape(min(kValRows, p.n_rows - rb));
  const int grp = w / sh.splits, split = w % sh.splits;
  const bool active = grp < sh.groups;
  const int r16 = rb + 16 * grp;
  uint32_t A[8][4];
  val_afrag([&](int i) { return active && r16 + i < p.n_rows ? val_row(p, ul, r16 + i) : nullptr; }, lane, A);
  const __nv_bfloat16* Ku = p.K + int64_t(ul) * p.s * kHeadDim;
  const __nv_bfloat16* Vu = p.V + int64_t(ul) * p.s * kHeadDim;
  const int32_t* top = p.top + int64_t(ul) * p.n_top;
  const int64_t e0 = int64_t(ul) * p.ent_stride + p.run_off[run];
  const int n_main = int((m + kTile - 1) / kTile), n = n_main + (r + kTile - 1) / kTile;
  auto issue = [&](int t) {                      // tile t into stage t & 1
    if (t < n) {
      const uint32_t dst = st_s + uint32_t((t & 1) * kValStage);
      float* bias = bias_s + (t & 1) * kTile;
      if (t < n_main) {
        const int64_t j0 = int64_t(t) * kTile;
        auto pos = [&](int i) -> int64_t {
          const int64_t j = j0 + i;
          return j >= m ? -1 : (j < keep ? top[j] : (p.s - p.recent) + (j - keep));
        };
        for (int idx = threadIdx.x; idx < kTile * 16; idx += kThreads) {
          const int row = idx >> 4, ch = idx & 15;
          const int64_t q = pos(row);
          const int64_t at = q < 0 ? 0 : q * kHeadDim + 8 * ch;
          cp_async16(dst + asg_swz(row, ch), Ku + at, q < 0 ? 0u : 16u);
          cp_async16(dst + kTile * kAsgRowBytes + asg_swz(row, ch), Vu + at, q < 0 ? 0u : 16u);
        }
        if (threadIdx.x < kTile) bias[threadIdx.x] = j0 + threadIdx.x < m ? 0.f : -INFINITY;
      } else {
        const int j0 = (t - n_main) * kTile;
        val_stage_rows(dst, [&](int i) { return j0 + i < r ? p.kbar + (e0 + j0 + i) * kHeadDim : nullptr; }, Ku);
        val_stage_rows(dst + kTile * kAsgRowBytes,
                       [&](int i) { return j0 + i < r ? p.vbar + (e0 + j0 + i) * kHeadDim : nullptr; }, Vu);
        if (threadIdx.x < kTile) {
          const int e = j0 + threadIdx.x;
          const int c = e < r ? p.ecount[e0 + e] : 0;       // an empty entry is inert
          bias[threadIdx.x] = c > 0 ? p.beta * logf(float(c)) * kLog2e : -INFINITY;
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float* my_rec = rec_m + w * 16 * kValRec;
  ValState st;
  st.reset();
  issue(0);
  for (int t = 0; t < n; ++t) {
    issue(t + 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (t == n_main && active) {                 // the residual branch begins
      val_store(st, [&](int i) { return my_rec + i * kValRec; });
      st.reset();
    }
    const uint32_t ks_s = st_s + uint32_t((t & 1) * kValStage);
    if (active) val_tile(st, A, ks_s, ks_s + kTile * kAsgRowBytes, split, sh.splits, bias_s + (t & 1) * kTile);
    __syncthreads();
  }
  if (active) {
    if (n == n_main) {                           // no residual entries
      val_store(st, [&](int i) { return my_rec + i * kValRec; });
      st.reset();
    }
    val_store(st, [&](int i) { return rec_r + (w * 16 + i) * kValRec; });
  }
  __syncthreads();
  // a warp per row: merge the splits of both branches, gate, error
  for (int i = w; i < 16 * sh.groups; i += kThreads / 32) {
    const int row = rb + i;
    if (row >= p.n_rows) break;
    float M[2], L[2];
    float4 acc[2];
#pragma unroll
    for (int br = 0; br < 2; ++br) {
      const float* rec = (br == 0 ? rec_m : rec_r) + ((i >> 4) * sh.splits * 16 + (i & 15)) * kValRec;
      float mx = -INFINITY, l = 0.f;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k = 0; k < sh.splits; ++k) mx = fmaxf(mx, rec[k * 16 * kValRec]);
      for (int k = 0; k < sh.splits; ++k) {
        const float* q = rec + k * 16 * kValRec;
        if (!(q[1] > 0.f)) continue;
        const float sc = exp2f(q[0] - mx);
        const float4 v = *reinterpret_cast<const float4*>(q + 4 + 4 * lane);
        l += q[1] * sc;
        a.x += v.x * sc;
        a.y += v.y * sc;
        a.z += v.z * sc;
        a.w += v.w * sc;
      }
      M[br] = mx;
      L[br] = l;
      acc[br] = a;
    }
    float g_val = p.g_fixed;
    if (p.gate_mode == RESKV_GATE_DYNAMIC) {
      const float pmax = 1.0f / L[0];            // M[0] is the largest main logit
      g_val = fmaxf(p.g_min, 1.0f / (1.0f + expf(-p.alpha * (p.tau - pmax))));
    }
    const float2 coef = branch_coefs(p.softmax_mode, g_val, M[0], L[0], M[1], L[1]);
    const float4 os = *reinterpret_cast<const float4*>(p.oS + (int64_t(ul) * p.n_rows + row) * kHeadDim + 4 * lane);
    const float dx = coef.x * acc[0].x + coef.y * acc[1].x - os.x, dy = coef.x * acc[0].y + coef.y * acc[1].y - os.y;
    const float dz = coef.x * acc[0].z + coef.y * acc[1].z - os.z, dw = coef.x * acc[0].w + coef.y * acc[1].w - os.w;
    const float e = warp_sum(dx * dx + dy * dy + dz * dz + dw * dw);
    if (lane == 0) p.rowerr[(int64_t(run) * p.UL + ul) * p.n_rows + row] = double(e);
  }
}

// L_r = mean of the per-query errors (fp64; a warp per unit and candidate); +inf
// for a unit without a candidate in this column (r = 0 in a column c > 0)
__global__ void k_loss_reduce(const double* rowerr, double* losses, int n_rows, int UL, int ncol,
                              const int32_t* r_runs) {
  const int i = int((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= UL * ncol) return;
  const int col = i / UL, ul = i % UL;
  const bool none = col > 0 && r_runs[i] == 0;
  double acc = 0.0;
  if (!none)
    for (int k = lane; k < n_rows; k += 32) acc += rowerr[int64_t(i) * n_rows + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) losses[int64_t(ul) * ncol + col] = none ? INFINITY : acc / double(n_rows);
}

// r* = argmin_{r>0} L_r (ties -> smaller r: columns hold ascending r); keep it
// only if L_r* < (1 - delta) L_0.  r_runs: [ncol, UL] r of every column.
__global__ void k_choose(const double* losses, int ncol, const int32_t* r_runs, int UL,
                         double one_minus_delta, int32_t* r_final, int32_t* chosen) {
  const int ul = blockIdx.x * blockDim.x + threadIdx.x;
  if (ul >= UL) return;
  const double* L = losses + int64_t(ul) * ncol;
  int best = 0;
  for (int c = 1; c < ncol; ++c)
    if (r_runs[int64_t(c) * UL + ul] > 0 && (best == 0 || L[c] < L[best])) best = c;
  const bool use = best > 0 && L[best] < one_minus_delta * L[0];
  r_final[ul] = use ? r_runs[int64_t(best) * UL + ul] : 0;
  chosen[ul] = use ? best : 0;
}

// ---------------------------------------------------------------------------
// Packing into the ragged layout (end of Alg. 1): main rows in position
// order, then the chosen run's residual entries.
// ---------------------------------------------------------------------------

struct PackArgs {
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  int64_t s;
  int32_t recent, budget;
  int32_t stride;              // slots per unit in the cache (budget + append capacity)
  const int32_t* rank_pos;     // [UL, s]
  const int32_t* r_final;      // [UL]
  const int32_t* chosen;       // [UL] run index of the chosen entries (0 = none)
  const int32_t* run_off;      // [n_runs] entry offset of each run
  const __nv_bfloat16* kbar;
  const __nv_bfloat16* vbar;
  const int32_t* ecount;
  int64_t ent_stride;
  float beta;
  int64_t unit0;               // global unit index of ul = 0
  __nv_bfloat16* kslots;
  __nv_bfloat16* vslots;
  float* logc;
  int32_t* slot_pos;
  int32_t* counts;
  int32_t* n_main;
  int32_t* n_res;
  const int32_t* budgets;      // [UL] per-unit budgets, or NULL (budget)
  const int32_t* offsets;      // [U + 1] first slot of every unit, or NULL (u * stride)
};

// One cluster per unit, as for the ranking: its CTAs take equal runs of
// positions, a warp 32 consecutive ones at a time, to list the main cache's in
// ascending order, then all warps of the cluster copy the rows.  What bounds it:
// the latency of few CTAs.  32 units of 128K keys, b = 2048: 27 us, 180 with one
// CTA per unit and a run of positions per thread; 64 units of 32K keys: 26, 63;
// 512 of 16K (one CTA each): 51, 59.
__global__ void __launch_bounds__(kTopThreads) k_pack(PackArgs p) {
  __shared__ int warp_sums[32];
  __shared__ int cta_total;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = int(cl.num_blocks()), rank = int(cl.block_rank());
  const int ul = blockIdx.x / cs;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t u = p.unit0 + ul;
  const int r = p.r_final[ul];
  const int64_t bu = unit_budget(p.budgets, ul, p.budget);
  const int64_t m = r == 0 ? (bu < p.s ? bu : p.s) : bu - r;
  const int64_t keep = m - p.recent;
  const int32_t* rp = p.rank_pos + int64_t(ul) * p.s;
  const int64_t base = p.offsets ? int64_t(p.offsets[u]) : u * p.stride;   // first slot of u
  int32_t* spos = p.slot_pos + base;
  // the warp's run of positions, a multiple of 32
  const int64_t run = (p.s + int64_t(cs) * kTopThreads - 1) / (int64_t(cs) * kTopThreads) * 32;
  const int64_t lo = (int64_t(rank) * (kTopThreads / 32) + w) * run, hi = lo + run < p.s ? lo + run : p.s;
  const int steps = lo < hi ? int((hi - lo + 31) >> 5) : 0;
  auto main_pos = [&](int64_t i, int32_t rk) { return i < hi && (rk < 0 || rk < keep); };
  unsigned saved = 0;                            // lane k: the bits of step k (of the first 32)
  int mine = 0;
  for (int k0 = 0; k0 < steps; k0 += 8) {        // eight loads in flight
    int32_t rk[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t i = lo + 32 * int64_t(k0 + k) + lane;
      rk[k] = i < hi ? __ldg(rp + i) : INT_MAX;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const unsigned f = __ballot_sync(0xffffffffu, main_pos(lo + 32 * int64_t(k0 + k) + lane, rk[k]));
      if (lane == k0 + k) saved = f;
      mine += __popc(f);
    }
  }
  if (lane == 0) warp_sums[w] = mine;
  __syncthreads();
  int out = 0;                                   // main positions before the warp's
  for (int k = 0; k < w; ++k) out += warp_sums[k];
  if (threadIdx.x == kTopThreads - 1) cta_total = out + mine;
  cl.sync();
  for (int k = 0; k < rank; ++k) out += *cl.map_shared_rank(&cta_total, k);
  for (int k = 0; k < steps; ++k) {
    const int64_t i = lo + 32 * int64_t(k);
    const unsigned f = k < 32 ? __shfl_sync(0xffffffffu, saved, k)
                              : __ballot_sync(0xffffffffu, main_pos(i + lane, i + lane < hi ? rp[i + lane] : INT_MAX));
    const int at = out + __popc(f & ((1u << lane) - 1u));
    if ((f >> lane & 1u) && at < m) spos[at] = int32_t(i + lane);
    out += __popc(f);
  }
  cl.sync();                                     // the list is complete (and cta_total read)
  const int w0 = rank * (kTopThreads / 32) + w, nw = cs * (kTopThreads / 32);
  const __nv_bfloat16* Ku = p.K + int64_t(ul) * p.s * kHeadDim;
  const __nv_bfloat16* Vu = p.V + int64_t(ul) * p.s * kHeadDim;
#pragma unroll 2
  for (int64_t j = w0; j < m; j += nw) {
    const int64_t pos = spos[j];
    const uint2 kw = __ldg(reinterpret_cast<const uint2*>(Ku + pos * kHeadDim) + lane);
    const uint2 vw = __ldg(reinterpret_cast<const uint2*>(Vu + pos * kHeadDim) + lane);
    reinterpret_cast<uint2*>(p.kslots + (base + j) * kHeadDim)[lane] = kw;
    reinterpret_cast<uint2*>(p.vslots + (base + j) * kHeadDim)[lane] = vw;
    if (lane == 0) {
      p.counts[base + j] = 0;
      p.logc[base + j] = 0.f;
    }
  }
  const int c = p.chosen[ul];
  for (int j = w0; j < r; j += nw) {
    const int64_t e = int64_t(ul) * p.ent_stride + p.run_off[c] + j;
    const int64_t slot = base + m + j;
    reinterpret_cast<uint2*>(p.kslots + slot * kHeadDim)[lane] =
        reinterpret_cast<const uint2*>(p.kbar + e * kHeadDim)[lane];
    reinterpret_cast<uint2*>(p.vslots + slot * kHeadDim)[lane] =
        reinterpret_cast<const uint2*>(p.vbar + e * kHeadDim)[lane];
    if (lane == 0) {
      const int cnt = p.ecount[e];
      p.counts[slot] = cnt;
      p.logc[slot] = cnt > 0 ? p.beta * logf(float(cnt)) : -INFINITY;
      spos[m + j] = -1;
    }
  }
  if (rank == 0 && threadIdx.x == 0) {
    p.n_main[u] = int32_t(m);
    p.n_res[u] = r;
  }
}

}  // namespace build
}  // namespace reskv
