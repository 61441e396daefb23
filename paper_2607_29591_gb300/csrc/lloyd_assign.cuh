// Lloyd assignment (Sec. 5.3, Eq. residual_partition) on the 5th-generation
// tensor cores: every evicted token to its nearest centre.
//
// The distances d_j = ||c_j||^2 - 2 <c_j, k> (the ||k||^2 term is common) need
// the dot products of every bf16 key with every centre.  Each fp32 centre is
// split exactly into two bf16 planes c = c1 + c2 + e, |e_i| <= 2^-16 |c_i|
// (split_planes), so <c, k> = <c1, k> + <c2, k> up to e: one tcgen05.mma chain
// per 128-token tile (2 planes x 8 K-steps of 16 dims, M = 128 tokens, N = r
// rounded up to 16) sums both planes in fp32 in tensor memory.
//
// k_lloyd_assign: a persistent CTA per SM walks a contiguous range of (unit,
// tile) pairs with the unit's planes resident in shared memory, so a tile costs
// one key-tile load and one MMA chain.  Four roles, linked by mbarriers:
//
//   loader warp      key tiles by TMA (both 64-dim halves, 128-byte swizzle,
//                    one 32 KB copy) into a ring of nk buffers, and the tokens'
//                    key norms and ranks by cp.async, as far ahead as the buffers
//                    allow, across unit changes too (key_full[]; a buffer is
//                    refilled once key_free[] says its MMAs are done).
//   2 MMA warps      warp b issues the MMA chains of the tiles t with t % 2 = b,
//                    into TMEM columns 256 b .., committed to full[b] and to the
//                    buffer's key_free[] (issuing a chain takes one warp about
//                    1300 cycles and its waits as many, more than a tile may
//                    take).  The warp with a unit's first tile waits until no MMA
//                    reads the old planes, then fetches the new ones and the
//                    centre norms by bulk copies (they lie in global memory as in
//                    shared).
//   16 column warps  warp w takes the tokens of TMEM lane quarter w % 4 and the
//                    16-column blocks w / 4, w / 4 + 4, ..: at most 64 distances
//                    of one token per thread, which stay in registers (the TMEM
//                    buffer is free as soon as they are there).  Two sweeps over
//                    them: the least, d0 (three-input minima); then the centres
//                    within W of it, as the sign bits of d_j - (d0 + W),
//                    funnel-shifted into words.  The candidates go to the
//                    deciders through shared memory (xch_full[], xch_free[]).
//   4 deciders       join the four column quarters' candidates of 32 tokens each
//                    and decide.
//
// W bounds what rounding can have moved (below), so a centre outside it cannot be
// nearest.  A token left with one centre is decided; the others (less than one per
// cent of centred keys) join a list of the CTA that k_lloyd_resolve decides exactly.
// The two sweeps take 1.5 integer-pipe operations per distance, where a running best
// three with packed indices took 6 and bounded the assignment.
//
// Units with more than 256 centres take their centres in segments of at most
// 256, one launch each: a launch leaves every token's least distance and
// candidates so far, the next one joins its own.
//
// A tile's steps are chains of dependent latencies, so what counts is how many
// warps work on different steps at once; 24 warps run with the registers moved
// (setmaxnreg) to the column warps.
//
// Tokens that joined and left a centre are counted in mcount by global
// reductions; where a unit has at most 64 centres, so that many tokens meet in
// one, each decider counts in shared memory and adds when it leaves the unit.
// Every wait is
// bounded; a wait that gives up raises kStatusWaitTimeout and an abort flag that
// ends every other wait.  No barrier is shared by warps that may leave.
//
// Error bound of a dot product, u = 2^-24, P = sum_i |c_i k_i|: one MMA step
// adds 16 exact products to the fp32 accumulator with an error of at most
// 17 * 2^-22 times the largest partial magnitude (<= P) even if it truncates to
// 24 bits; 16 chained steps (both planes) give 272 * 2^-22 P = 1088u P, the split
// e adds 256u P, |c1| + |c2| exceeds |c| by 2^-8: 1350u P, taken as 1440u P.  (A
// bound three times as wide cost k_lloyd_resolve 1.7 to 2.1 times its time.  Measured
// on GB300 over 43 kinds of rows -- one sign, one product far above the others in a
// step or in the chain, cancelling ones, every alignment to the accumulator -- a chain
// was never more than 45u P off where 1088u P is allowed.)
// Values, products and sums below 2^-126 may be lost besides, whole at worst: 2^-126
// sum_i (|c_i| + |k_i|) <= 12 * 2^-126 (||c|| + ||k||) for the operands, twice that in a
// distance, and some 600 terms of 2^-126.  The bounds of both norms are kNormLost =
// 2^-50 above them, which adds 2^-62 (||c|| + ||k||) + 2^-112 to W's dot products: more
// than all of that.  So W is positive however small the distances are, and centres
// at equal ones (all of them zero, say) are candidates.
//
// What bounds it: issue and the latency of a tile's steps (about 2.3 instructions
// per cycle; the tensor pipe is active 27 % of the time at r = 51 and 54 % at 204,
// DRAM 66 % and 41 %).  64 units of 32K keys (16384 tiles) take 112, 129, 149 and
// 177 us at r = 51, 102, 153, 204; the running best three took 148, 180, 221 and
// 265.  32 units of 128K keys at r = 409 take 685 us in two segments, where a
// kernel that streamed the centres per tile took 4500.
// Tried and slower: 2 x 4 column warps with 32-column loads (141 to 310 us), 2 x 8
// that read TMEM twice (139 to 186), and deciding in the column warps, in turn or
// by one quarter (133 to 208).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "construct_kernels.cuh"

namespace reskv {
namespace build {

constexpr int kAsgColWarps = 16;
constexpr int kAsgDecide = kAsgColWarps;                        // the first decider's index
constexpr int kAsgMma = kAsgDecide + 4;                         // the first MMA-issuing warp's index
constexpr int kAsgLoader = kAsgMma + 2;                         // the key-loading warp's index
constexpr int kAsgThreads = (kAsgLoader + 2) * 32;              // (one warp idle: whole warpgroups)
// Registers a thread: 80 at launch (24 warps of the SM's 65,536), then 88 for the
// 16 column warps and 56 for the other 8: 512 x 88 + 256 x 56 <= 768 x 80.
constexpr int kAsgRegsCol = 88, kAsgRegsOther = 56;
static_assert(kAsgColWarps * kAsgRegsCol + (kAsgThreads / 32 - kAsgColWarps) * kAsgRegsOther <=
                  (kAsgThreads / 32) * 80,
              "setmaxnreg must not ask for more than the launch holds");
constexpr int kAsgRmax = 256;                                   // centres of one segment
constexpr int kAsgCnt = 64;                                     // centres counted in shared memory, at most
constexpr int kTcHalf = kTile * 128;                            // one 64-dim half of a key tile, bytes
constexpr int kAsgKeys = 2 * kTcHalf;                           // one key tile
constexpr uint32_t kAsgBufCols = 256;                           // TMEM columns per buffer
constexpr uint32_t kAsgCols = 2 * kAsgBufCols;
constexpr int kAsgMaxKeyBufs = 4;
// Tiles whose key norms and ranks are held: the loader is at most nk tiles past
// the last tile whose MMAs are done, and those are at most 2 tiles past the last
// one the column warps have read.
constexpr int kAsgInfo = 8;
static_assert(kAsgInfo >= kAsgMaxKeyBufs + 3, "a tile's norms must outlive its readers");
constexpr long long kTcWaitCycles = 4000000000LL;

// Dynamic shared memory, from a 1024-aligned base: the planes of rp = r rounded
// up to 16 centres ([plane][64-dim half][rp rows][128 B], 512 rp bytes) and nk
// key tiles of 32 KB.  The small parts are static, so that their addresses cost
// no registers: the column warps hold 64 distances in their 88 registers
// (kAsgRegsCol), and what spilled would not fit the L1 beside 220 KB.
struct AsgShared {
  float cn[2][kAsgRmax];                               // centre norms (two units)
  int2 xch[2][4][kTile];                               // the column quarters' candidates (two tiles)
  float xw[2][kTile];                                  // the tokens' windows
  int xrk[2][kTile];                                   // and ranks
  float kn[kAsgInfo][kTile];                           // the tile's key norms and ranks
  int rk[kAsgInfo][kTile];
  int cnt[4][2][kAsgCnt];                              // the deciders' counts: joined, left
  int tinfo[2][2];                                     // per TMEM buffer: max ||c||, norm buffer
  uint32_t abort;
  int amb_n;                                           // listed tokens
  uint64_t full[2];                                    // MMA commit + the MMA warp
  uint64_t tmem_empty[2];                              // column warps
  uint64_t xch_full[2];                                // column warps
  uint64_t xch_free[2];                                // deciders
  uint64_t planes_full;                                // planes and norms of a unit
  uint64_t key_full[kAsgMaxKeyBufs];                   // the key tile's bytes
  uint64_t key_free[kAsgMaxKeyBufs];                   // MMA commit: buffer read
  uint32_t tmem;                                       // TMEM address
};
constexpr size_t kAsgSmemMax = 232448 - ((sizeof(AsgShared) + 1023) & ~size_t(1023));   // of 227 KB per CTA

__host__ __device__ inline size_t lloyd_asg_planes(int rp) { return size_t(rp) * 512; }
// key buffers that fit beside the planes of rp centres (>= 2 for rp <= 256)
inline int lloyd_asg_key_bufs(int rp) {
  return int(std::min<size_t>(kAsgMaxKeyBufs, (kAsgSmemMax - 1024 - lloyd_asg_planes(rp)) / kAsgKeys));
}
inline size_t lloyd_asg_smem(int rp) {
  return 1024 + lloyd_asg_planes(rp) + size_t(lloyd_asg_key_bufs(rp)) * kAsgKeys;
}

// Shared-memory matrix descriptor: start address (16-byte units), leading
// byte offset 1 (unused by swizzled K-major layouts), stride byte offset
// 1024 (8-row groups), descriptor version 1, 128-byte swizzle.  Operands are
// K-major: per 64-dim half, rows of 128 bytes, the 16-byte chunk c of row r at
// ((c ^ (r & 7)) << 4); the K-steps inside a half advance the start by 32 bytes.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return uint64_t((saddr & 0x3FFFFu) >> 4) | (uint64_t(1) << 16) | (uint64_t(1024 >> 4) << 32) |
         (uint64_t(1) << 46) | (uint64_t(2) << 61);
}

// A shared-memory descriptor advanced by `bytes` (a multiple of 16): the start
// address sits in bits 0..13 as address / 16, and stays below 2^14 for the
// 227 KB of shared memory, so the low word takes the addition without carry.
__device__ __forceinline__ uint64_t desc_plus(uint64_t d, uint32_t bytes) {
  return d + uint64_t(bytes >> 4);
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, M = 128, N = n (a multiple of 16, <= 256).
__device__ __forceinline__ uint32_t tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(n >> 3) << 17) | (uint32_t(kTile >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc,
                                       bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate ? 1 : 0));
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane from column address
// ta, there after tc_ld_wait
__device__ __forceinline__ void tc_ld16(uint32_t ta, float* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15}, [%16];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
        "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]),
        "=f"(r[15])
      : "r"(ta));
}

// waits for the warp's TMEM loads; the 16 values are defined from here on
__device__ __forceinline__ void tc_ld_wait(float* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]),
                 "+f"(r[7]), "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]), "+f"(r[12]), "+f"(r[13]),
                 "+f"(r[14]), "+f"(r[15])
               :
               : "memory");
}

// one 128-token key tile (both 64-dim halves, 128-byte swizzle) from row y
// of the layer's keys, completing on bar
__device__ __forceinline__ void tma_keys(uint32_t dst, const CUtensorMap* map, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(y), "r"(0), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// One arrival for the warp, after everything its lanes did before (an arrival
// per thread is serialised in shared memory: 512 of them took longer than a
// tile's MMAs).
__device__ __forceinline__ void asg_arrive(uint64_t* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Wait for phase `parity` of bar; false after the bound or once the abort
// flag is up.
__device__ __forceinline__ bool asg_wait(uint64_t* bar, uint32_t parity, const volatile uint32_t* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort != 0u || clock64() - t0 > kTcWaitCycles) return false;
  }
  return true;
}

__device__ __forceinline__ void asg_raise(volatile uint32_t* abort, uint32_t* status) {
  if (*abort == 0u) {
    *abort = 1u;
    report_status(status, kStatusWaitTimeout);
  }
}

// the least of three (one instruction on sm_100 and later); NaN operands lose
__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// m shifted left by one, the sign bit of x coming in
__device__ __forceinline__ uint32_t push_sign(uint32_t m, float x) {
  uint32_t d;
  asm("shf.l.wrap.b32 %0, %1, %2, 1;" : "=r"(d) : "r"(__float_as_uint(x)), "r"(m));
  return d;
}

// (unit, tile) of the flat tile order g = unit * ntiles + tile, stepped without
// divisions, skipping units with no centre from seg0 on; r is read once per unit
struct AsgCursor {
  int g, u, tile, r;
  __device__ AsgCursor(const LloydArgs& p, int g0, int g1, int seg0) : g(g0) {
    u = g0 / p.ntiles;
    tile = g0 - u * p.ntiles;
    r = g < g1 ? p.r_unit[u] : 0;
    skip(p, g1, seg0);
  }
  __device__ void skip(const LloydArgs& p, int g1, int seg0) {
    while (g < g1 && r <= seg0) {
      g += p.ntiles - tile;
      tile = 0;
      ++u;
      r = g < g1 ? p.r_unit[u] : 0;
    }
  }
  __device__ void next(const LloydArgs& p, int g1, int seg0) {
    ++g;
    if (++tile == p.ntiles) {
      tile = 0;
      ++u;
      r = g < g1 ? p.r_unit[u] : 0;
    }
    skip(p, g1, seg0);
  }
};

// How far from a distance d a centre's distance may lie while it could still be
// nearest; ww: the part that does not depend on d.
__device__ __forceinline__ float asg_window(float ww, float d) { return ww + 10.0f * 5.9604645e-8f * fabsf(d); }

// The candidates of a token: the least distance, the first and last candidate
// (centre indices below 2^14) and how many there are (1, 2, or 3 for more).
struct AsgCand {
  float d;
  int first, last, n;
  __device__ __forceinline__ int2 pack() const {
    return make_int2(__float_as_int(d), first | (last << 14) | (n << 28));
  }
  __device__ static __forceinline__ AsgCand unpack(int2 v) {
    return AsgCand{__int_as_float(v.x), v.y & 0x3fff, (v.y >> 14) & 0x3fff, (v.y >> 28) & 3};
  }
};

// The tiles [g0, g1) of the flat (unit, tile) order, g = unit * ntiles + tile,
// against the centres [seg0, seg0 + segw) of each unit (segw <= 256, a multiple
// of 16; units with fewer centres are skipped).  The launch that sees a unit's
// last centre decides its tokens: assign (centre index, -1 for tokens outside
// E), the counts of moves (mcount), and the list of tokens left (amb: the CTA's
// entries from tile g0's place on, amb_count).  p.knorm holds the key norms.
// NB: 16-column blocks per column warp, segw <= 64 NB.
template <int NB>
__global__ void __launch_bounds__(kAsgThreads, 1)
    k_lloyd_assign(LloydArgs p, int seg0, int segw, int nk, const __grid_constant__ CUtensorMap tmK) {
  extern __shared__ uint8_t asg_raw[];
  uint8_t* base = asg_raw + ((1024u - (smem_u32(asg_raw) & 1023u)) & 1023u);
  const uint32_t plane_half = uint32_t(segw) * 128u;             // one plane's 64-dim half, bytes
  __shared__ __align__(16) AsgShared sh;
  const uint32_t planes_s = smem_u32(base), keys_s = planes_s + uint32_t(lloyd_asg_planes(segw));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n_all = int64_t(p.n_units) * p.ntiles;   // below 2^31 (the tokens are)
  const int g0 = int(n_all * blockIdx.x / gridDim.x), g1 = int(n_all * (blockIdx.x + 1) / gridDim.x);

  for (int i = tid; i < 8 * kAsgCnt; i += kAsgThreads) sh.cnt[0][0][i] = 0;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.full[i], 2);
      mbar_init(&sh.tmem_empty[i], kAsgColWarps);
      mbar_init(&sh.xch_full[i], kAsgColWarps);
      mbar_init(&sh.xch_free[i], 4);
    }
    mbar_init(&sh.planes_full, 1);
    for (int i = 0; i < nk; ++i) {
      mbar_init(&sh.key_full[i], 33);       // the key tile's bytes, every lane's cp.async
      mbar_init(&sh.key_free[i], 1);
    }
    sh.abort = 0u;
    sh.amb_n = seg0 == 0 ? 0 : p.amb_count[blockIdx.x];   // later segments go on with the list
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                 "r"(kAsgCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem;

  if (warp < kAsgColWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kAsgRegsCol));
    // ---------------- column warps ----------------
    const int quarter = warp >> 2, q = warp & 3, tok = 32 * q + lane;
    const uint32_t tb = tmem + (uint32_t(32 * q) << 16);
    int t = 0;
    bool ok = true;
    for (AsgCursor cc(p, g0, g1, seg0); cc.g < g1; cc.next(p, g1, seg0)) {
      const int b = t & 1;
      ok = asg_wait(&sh.full[b], uint32_t((t >> 1) & 1), &sh.abort);
      if (p.test_fault && blockIdx.x == 0 && t == 0) ok = false;   // a timed-out wait, injected
      if (__any_sync(0xffffffffu, !ok)) break;
      tc_fence_after();
      const float cm = __int_as_float(sh.tinfo[b][0]), kn = sh.kn[t % kAsgInfo][tok];
      const int rk = sh.rk[t % kAsgInfo][tok];          // taken on by quarter 0
      const float* cn = sh.cn[sh.tinfo[b][1]];
      // the token's distances to the centres seg0 + 16 (quarter + 4 i) + 0..15.
      // A column past the unit's centres holds anything; its norm is +inf, so
      // its distance is +inf or NaN and neither sweep takes it.  (Loading under
      // a condition instead made the registers spill.)
      float d[NB][16];
#pragma unroll
      for (int i = 0; i < NB; ++i)
        tc_ld16(tb + uint32_t(b) * kAsgBufCols + uint32_t(16 * (quarter + 4 * i)), d[i]);
      float a[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        tc_ld_wait(d[i]);
        const float2 m2 = make_float2(-2.0f, -2.0f);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const float4 n = *reinterpret_cast<const float4*>(cn + 16 * (quarter + 4 * i) + 4 * x);
          float* dx = d[i] + 4 * x;
          const float2 lo = ffma2(m2, make_float2(dx[0], dx[1]), make_float2(n.x, n.y));
          const float2 hi = ffma2(m2, make_float2(dx[2], dx[3]), make_float2(n.z, n.w));
          dx[0] = lo.x;
          dx[1] = lo.y;
          dx[2] = hi.x;
          dx[3] = hi.y;
          a[x] = min3(min3(a[x], lo.x, lo.y), hi.x, hi.y);
        }
      }
      tc_fence_before();
      asg_arrive(&sh.tmem_empty[b]);                         // TMEM buffer, tile info and norms are free
      const float d0 = fminf(min3(a[0], a[1], a[2]), a[3]);
      // A computed distance is off by at most ee + 4u |d| from the exact distance
      // to the fp64 centre: ee = 2 x dot product (gam_tc ||c|| ||k||, and 2u for
      // the fp32 centre) + norm sum gam ||c||^2 (130u, and 2u for the fp32 centre),
      // ||c|| <= max ||c|| over the unit.  So the nearest centre's computed
      // distance is within 2 ee + 4u (|d0| + |d|) of d0.
      const float uu = 5.9604645e-8f, gam = 140.0f * uu, gam_tc = 1440.0f * uu;
      const float ee = cm * (2.0f * gam_tc * kn + gam * cm);
      const float ww = 2.01f * ee;
      const float thr = d0 + asg_window(ww, d0);
      const float2 nthr = make_float2(-thr, -thr);
      uint32_t m[2] = {0u, 0u};                           // two blocks each, first column in the high bit
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int x = 0; x < 4; x += 2) {
            const float2 e = fadd2(make_float2(d[i][4 * y + x], d[i][4 * y + x + 1]), nthr);
            w[y] = push_sign(push_sign(w[y], e.x), e.y);
          }
        const uint32_t v = (((w[0] << 4) | w[1]) << 8) | (w[2] << 4) | w[3];
        m[i >> 1] |= (i & 1) ? v : v << 16;
      }
      AsgCand cd{d0, 0, 0, min(__popc(m[0]) + __popc(m[1]), 3)};
      if (cd.n != 0) {                                    // (else no centre, or NaN or infinite distances)
        const int pf = m[0] != 0u ? __clz(m[0]) : 32 + __clz(m[1]);
        const int pl = m[1] != 0u ? 64 - __ffs(m[1]) : 32 - __ffs(m[0]);
        cd.first = seg0 + 16 * quarter + (pf & 15) + ((pf & 48) << 2);
        cd.last = seg0 + 16 * quarter + (pl & 15) + ((pl & 48) << 2);
      }
      ok = t < 2 || asg_wait(&sh.xch_free[b], uint32_t(((t >> 1) - 1) & 1), &sh.abort);
      if (__any_sync(0xffffffffu, !ok)) break;
      sh.xch[b][quarter][tok] = cd.pack();
      if (quarter == 0) {
        sh.xw[b][tok] = ww;
        sh.xrk[b][tok] = rk;
      }
      asg_arrive(&sh.xch_full[b]);
      ++t;
    }
    if (!ok) asg_raise(&sh.abort, p.status);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kAsgRegsOther));
    if (warp == kAsgLoader) {
      // ---------------- loader ----------------
      int nl = 0;
      bool ok = true;
      for (AsgCursor cl(p, g0, g1, seg0); cl.g < g1; cl.next(p, g1, seg0), ++nl) {
        const int slot = nl % nk;
        if (nl >= nk) {                                // MMA(nl - nk) has read the buffer
          const bool w = asg_wait(&sh.key_free[slot], uint32_t(((nl / nk) - 1) & 1), &sh.abort);
          if (__any_sync(0xffffffffu, !w)) {
            ok = false;
            break;
          }
        }
        if (lane == 0) {
          mbar_arrive_expect_tx(&sh.key_full[slot], uint32_t(kAsgKeys));
          tma_keys(keys_s + uint32_t(slot * kAsgKeys), &tmK,
                   int(int64_t(cl.u % p.UL) * p.s + int64_t(cl.tile) * kTile), &sh.key_full[slot]);
        }
        const int64_t row0 = int64_t(cl.u % p.UL) * p.s;
  #pragma unroll
        for (int i = lane; i < kTile; i += 32) {
          const int64_t pos = int64_t(cl.tile) * kTile + i;
          if (pos < p.s) {
            cp_async4(smem_u32(&sh.kn[nl % kAsgInfo][i]), p.knorm + row0 + pos);
            cp_async4(smem_u32(&sh.rk[nl % kAsgInfo][i]), p.rank_pos + row0 + pos);
          }
        }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&sh.key_full[slot])) : "memory");
        // the candidates and the centres so far into L2, a line a lane
        const int64_t t0 = int64_t(cl.tile) * kTile + (lane < 8 ? 16 * lane : 32 * (lane & 3));
        if (t0 < p.s) {
          if (lane < 8 && seg0 > 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.cand + int64_t(cl.u) * p.s + t0));
          if (lane >= 8 && lane < 12 && p.assign_prev)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.assign_prev + int64_t(cl.u) * p.s + t0));
        }
      }
      if (!ok && lane == 0) asg_raise(&sh.abort, p.status);
      // the copies in flight land before the CTA exits (the latest phase of
      // each buffer: no older one can alias it)
      const long long t0 = clock64();
      for (int i = nl > nk ? nl - nk : 0; i < nl; ++i)
        while (!mbar_try_wait(&sh.key_full[i % nk], uint32_t((i / nk) & 1)) && clock64() - t0 < kTcWaitCycles) {
        }
    } else if (warp == kAsgMma || warp == kAsgMma + 1) {
      // ---------------- MMA issue ----------------
      const int bb = warp - kAsgMma;                   // the TMEM buffer and the parity of its tiles
      int nm = 0, cur_u = -1, nu = 0;                  // tiles and units so far
      float cmx = 0.f;                                 // max ||c|| of the unit
      bool ok = true, planes_pending = false;
      int nu_seen = 0, last = -1;                      // the planes waited for; the last tile issued
      const uint64_t da0 = tc_desc(keys_s), db0 = tc_desc(planes_s);   // descriptors of the bases
      for (AsgCursor cm(p, g0, g1, seg0); cm.g < g1; cm.next(p, g1, seg0), ++nm) {
        const int u = cm.u, rs = min(cm.r - seg0, segw), rpad = (rs + 15) & ~15;
        const bool first = u != cur_u;
        if (first) ++nu;                               // this unit's planes and norms: load number nu - 1
        cur_u = u;
        if ((nm & 1) != bb) continue;
        if (first) {
          // no MMA reads the old planes once the last two tiles' are done; the
          // norms go to the other buffer, which the tile before the last read
          // last.  The columns' wait comes first: they are done with tile nm - 2,
          // so with nm - 3, so the other warp's barrier is in the phase of tile
          // nm - 1 or past it and its parity tells them apart.
          if (nm >= 1) {
            bool w = (nm < 2 || asg_wait(&sh.tmem_empty[bb], uint32_t(((nm - 2) >> 1) & 1), &sh.abort)) &&
                     asg_wait(&sh.full[bb ^ 1], uint32_t(((nm - 1) >> 1) & 1), &sh.abort);
            if (__any_sync(0xffffffffu, !w)) {
              ok = false;
              break;
            }
          }
          const int64_t c0 = int64_t(u) * p.rmax;
          for (int i = rpad + lane; i < kAsgRmax; i += 32) sh.cn[(nu - 1) & 1][i] = INFINITY;
          __syncwarp();
          if (lane == 0) {
            mbar_arrive_expect_tx(&sh.planes_full, uint32_t(rpad) * (4u * 128u + 4u));
            const uint8_t* src = reinterpret_cast<const uint8_t*>(p.cplanes) + (c0 * 4 + seg0) * 128;
            for (int ph = 0; ph < 4; ++ph)
              bulk_g2s(base + uint32_t(ph) * plane_half, src + int64_t(ph) * p.rmax * 128, uint32_t(rpad) * 128u,
                       &sh.planes_full);
            bulk_g2s(sh.cn[(nu - 1) & 1], p.cnorm + c0 + seg0, uint32_t(rpad) * 4u, &sh.planes_full);
          }
          planes_pending = true;
        }
        if (nu != nu_seen) {                           // the unit's first tile of this warp
          const int64_t c0 = int64_t(u) * p.rmax;
          cmx = 0.f;
          for (int i = lane; i < cm.r; i += 32) cmx = fmaxf(cmx, p.cnorm[c0 + i]);
  #pragma unroll
          for (int o = 16; o > 0; o >>= 1) cmx = fmaxf(cmx, __shfl_xor_sync(0xffffffffu, cmx, o));
          cmx = sqrtf(cmx) + kNormLost;
          const bool w = asg_wait(&sh.planes_full, uint32_t((nu - 1) & 1), &sh.abort);
          if (__any_sync(0xffffffffu, !w)) {
            ok = false;
            break;
          }
          planes_pending = false;
          nu_seen = nu;
        }
        // tile nm: a free TMEM buffer, its keys, then the MMA chain.  (In this
        // order: with 3 key buffers the slot's previous tile nm - 3 is the other
        // warp's, and the columns being done with tile nm - 2 says that it has
        // arrived, so that the slot's parity is that of tile nm.)
        const int slot = nm % nk;
        bool w = (nm < 2 || asg_wait(&sh.tmem_empty[bb], uint32_t(((nm - 2) >> 1) & 1), &sh.abort)) &&
                 asg_wait(&sh.key_full[slot], uint32_t((nm / nk) & 1), &sh.abort);
        if (__any_sync(0xffffffffu, !w)) {
          ok = false;
          break;
        }
        __syncwarp();
        if (lane == 0) {
          sh.tinfo[bb][0] = __float_as_int(cmx);
          sh.tinfo[bb][1] = (nu - 1) & 1;
          tc_fence_after();
          const uint32_t idesc = tc_idesc(rpad);
          const uint32_t d_tmem = tmem + uint32_t(bb) * kAsgBufCols;
          const uint64_t da = desc_plus(da0, uint32_t(slot * kAsgKeys));
  #pragma unroll
          for (int pl = 0; pl < 2; ++pl)
  #pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint32_t half = uint32_t(k >> 2), kk = uint32_t(k & 3) * 32u;
              tc_mma(d_tmem, desc_plus(da, half * kTcHalf + kk),
                     desc_plus(db0, uint32_t(pl * 2 + half) * plane_half + kk), idesc, pl + k > 0);
            }
          tc_commit(&sh.full[bb]);
          tc_commit(&sh.key_free[slot]);
        }
        asg_arrive(&sh.full[bb]);
        last = nm;
      }
      if (!ok && lane == 0) asg_raise(&sh.abort, p.status);
      // every copy has landed and every issued MMA is done before TMEM is freed
      const long long t0 = clock64();
      if (planes_pending)
        while (!mbar_try_wait(&sh.planes_full, uint32_t((nu - 1) & 1)) && clock64() - t0 < kTcWaitCycles) {
        }
      if (last >= 0)
        while (!mbar_try_wait(&sh.full[bb], uint32_t((last >> 1) & 1)) && clock64() - t0 < kTcWaitCycles) {
        }
    } else if (warp < kAsgMma) {
      // ---------------- deciders ----------------
      const int q = warp - kAsgDecide, tok = 32 * q + lane;
      int t = 0, cur_u = -1, keep = 0;
      // the warp's counts of the unit so far into mcount
      auto flush = [&]() {
        __syncwarp();
        if (cur_u >= 0 && p.r_unit[cur_u] <= kAsgCnt)
          for (int i = lane; i < 2 * kAsgCnt; i += 32) {
            const int h = i / kAsgCnt, j = i % kAsgCnt, c = sh.cnt[q][h][j];
            if (c != 0) atomicAdd(p.mcount + (2 * int64_t(cur_u) + h) * p.rmax + j, c);
            sh.cnt[q][h][j] = 0;
          }
        __syncwarp();
      };
      bool ok = true;
      for (AsgCursor cc(p, g0, g1, seg0); cc.g < g1; cc.next(p, g1, seg0), ++t) {
        const int u = cc.u, r = cc.r, b = t & 1, pos = cc.tile * kTile + tok;
        const bool mine = pos < p.s;
        if (u != cur_u) {
          flush();
          cur_u = u;
          keep = int(unit_budget(p.budgets, u % p.UL, p.budget)) - r - p.recent;   // ranked tokens from here on are in E
        }
        const int64_t tix = int64_t(u) * p.s + pos;
        const int old = mine && p.assign_prev ? p.assign_prev[tix] : -1;   // (in L2 by now)
        ok = asg_wait(&sh.xch_full[b], uint32_t((t >> 1) & 1), &sh.abort);
        if (__any_sync(0xffffffffu, !ok)) break;
        const float ww = sh.xw[b][tok];
        const int rk = sh.xrk[b][tok];
        const int2 x0 = sh.xch[b][0][tok], x1 = sh.xch[b][1][tok], x2 = sh.xch[b][2][tok], x3 = sh.xch[b][3][tok];
        asg_arrive(&sh.xch_free[b]);
        // the candidates of two sets of centres together
        auto join = [&](const AsgCand& v, const AsgCand& w) {
          if (v.n == 0 || w.d + asg_window(ww, w.d) < v.d) return w;
          if (w.n == 0 || v.d + asg_window(ww, v.d) < w.d) return v;
          return AsgCand{fminf(v.d, w.d), min(v.first, w.first), max(v.last, w.last), v.n + w.n > 2 ? 3 : 2};
        };
        AsgCand cd = join(AsgCand::unpack(x0), AsgCand::unpack(x1));
        cd = join(cd, AsgCand::unpack(x2));
        cd = join(cd, AsgCand::unpack(x3));
        // Below a window of 1e32 every product, sum and norm is finite.  Past it a
        // centre may lie beside the token at a distance that overflowed, so all
        // centres are candidates (where any distance is a number below infinity).
        if (!(ww < 1e32f)) {
          const float d = fminf(min3(__int_as_float(x0.x), __int_as_float(x1.x), __int_as_float(x2.x)), __int_as_float(x3.x));
          cd = AsgCand{d, 0, 0, d < INFINITY ? 3 : 0};
        }
        if (seg0 > 0 && mine) cd = join(AsgCand::unpack(p.cand[tix]), cd);   // the segments before
        if (r > seg0 + segw) {                              // more centres in the next launch
          if (mine) p.cand[tix] = cd.pack();
          continue;
        }
        const bool ev = mine && rk >= 0 && rk >= keep;       // in E (in_evicted)
        if (ev && cd.n == 0) {
          report_status(p.status, kStatusBadIndex);
          cd = AsgCand{0.f, 0, 0, 1};
        }
        const bool listed = ev && cd.n > 1;
        const unsigned bal = __ballot_sync(0xffffffffu, listed);
        if (bal != 0u) {
          int at = 0;
          if (lane == 0) at = atomicAdd(&sh.amb_n, __popc(bal));
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
          if (listed)
            p.amb[int64_t(g0) * kTile + at] = make_int4(u, pos, cd.first | (cd.n > 2 ? int(0x80000000u) : 0), cd.last);
        }
        if (listed) {
          // decided, written and counted by k_lloyd_resolve
        } else if (ev) {
          p.assign[tix] = cd.first;
          if (cd.first != old) {
            const int64_t c0 = 2 * int64_t(u) * p.rmax;
            if (r <= kAsgCnt) {
              atomicAdd(&sh.cnt[q][0][cd.first], 1);
              if (old >= 0) atomicAdd(&sh.cnt[q][1][min(old, kAsgCnt - 1)], 1);
            } else {
              atomicAdd(p.mcount + c0 + cd.first, 1);
              if (old >= 0) atomicAdd(p.mcount + c0 + p.rmax + min(old, r - 1), 1);
            }
          }
        } else if (mine) {
          p.assign[tix] = -1;
        }
      }
      if (!ok) asg_raise(&sh.abort, p.status);
      flush();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0) p.amb_count[blockIdx.x] = sh.amb_n;
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAsgCols));
  }
}

// The decision of the tokens k_lloyd_assign left.  Candidates: the two kept
// centres (nearly always), or every centre when more were within the tensor-core
// bound.  A warp takes four tokens of two candidates at once, eight lanes each
// (lane l on dims 4l + 32i .. 4l + 32i + 3, i < 4).  The tokens of all centres
// that the CTA met are queued and their distances shared out over its warps (lane
// l on dims 4l .. 4l + 3), then a warp per token decides.  A distance is the same
// tree of sums either way: chains of 4 dims, then dims 64, 32, 16, 8 and 4 apart.
// Bound by latency: 0.3 to 0.9 % of the tokens come here, one in a hundred of them
// with all centres, whose serial scan by one warp used to end the kernel.  64
// units of 32K keys, r = 51 .. 205: 18 us on average, 34 with a warp per token of
// either kind; 32 units of 128K keys, r = 102 .. 410: 34, 67.
//
// First their distances are taken directly in fp32, d32_j = sum_i (k_i -
// c32_i)^2 against the fp32 centres: no cancellation, so the error is small
// relative to the distance itself.  With u = 2^-24, |d32_j - D_j| <= b_j =
// 16 u d32_j + 3 u ||c_j|| (sqrt(d32_j) + u ||c_j||) bounds the difference to
// the exact distance D_j to the fp64 centre (12 u for the rounded differences,
// the 4-term chain and the 5 butterfly levels; 2 u ||c|| (2 sqrt(D) + u ||c||)
// for |c32 - c64| <= u ||c||; the rest is slack for using d32 in place of D); 2^-126
// is added, far more than squares that underflow can lose.
// The fp32 best decides unless another candidate's interval
// [d32_j - b_j, d32_j + b_j] reaches the best's; those few are re-evaluated in
// fp64, ties to the lower index.  Writes assign and counts the move.
constexpr int kResWarps = 8;
constexpr int kResChunk = 256;                  // distances held at once
constexpr int kResMaxCtas = 1024;               // assignment CTAs (one list each)

__global__ void __launch_bounds__(kResWarps * 32, 3) k_lloyd_resolve(LloydArgs p, int n_lists) {
  __shared__ float dsm[kResWarps][kResChunk];     // candidate distances (fp32) of kResWarps queued tokens
  __shared__ int jsm[kResWarps][kResChunk];       // centres left for fp64
  __shared__ int2 queue[4 * kResWarps];           // (unit, position) of the tokens of all centres
  __shared__ int queued;
  __shared__ int pre[kResMaxCtas + 1];            // tokens in the lists before list i
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
  float* dl = dsm[wb];
  int* jl = jsm[wb];
  {
    const int per = (n_lists + blockDim.x - 1) / blockDim.x, i0 = threadIdx.x * per;
    int mine = 0;
    for (int i = i0; i < min(i0 + per, n_lists); ++i) mine += p.amb_count[i];
    int total = 0;
    int run = block_exclusive_scan(mine, warp_sums, &total);
    for (int i = i0; i < min(i0 + per, n_lists); ++i) {
      pre[i] = run;
      run += p.amb_count[i];
    }
    if (threadIdx.x == 0) {
      pre[n_lists] = total;
      queued = 0;
    }
    __syncthreads();
  }
  const int n = pre[n_lists];
  const int64_t n_all = int64_t(p.n_units) * p.ntiles;
  const int nw = int((int64_t(gridDim.x) * blockDim.x) >> 5);
  const float uu = 5.9604645e-8f;
  // the decision res (>= r: none, only NaN distances get there)
  auto settle = [&](int u, int r, int64_t pos, int res) {
    if (res >= r) {
      report_status(p.status, kStatusBadIndex);
      res = 0;
    }
    p.assign[int64_t(u) * p.s + pos] = res;
    const int old = p.assign_prev ? p.assign_prev[int64_t(u) * p.s + pos] : -1;
    if (res != old) {
      atomicAdd(p.mcount + 2 * int64_t(u) * p.rmax + res, 1);
      if (old >= 0) atomicAdd(p.mcount + (2 * int64_t(u) + 1) * p.rmax + min(old, r - 1), 1);
    }
  };
  auto interval = [&](float d, float norm2) {
    const float cn = sqrtf(norm2) * 1.001f;
    return 16.0f * uu * d + 3.0f * uu * cn * (sqrtf(d) + uu * cn) + FLT_MIN;
  };
  // (four tokens nw apart: where there are few, every warp has one at most)
  for (int64_t i0 = 0; i0 < n; i0 += 4 * nw) {
    const int64_t i = i0 + ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) + int64_t(lane >> 3) * nw;
    const int c8 = lane & 7;
    int4 e = make_int4(0, 0, 0, 0);
    if (i < n) {
      int li = 0, hi_l = n_lists;                 // the list holding token i
      while (hi_l - li > 1) {
        const int mid = (li + hi_l) >> 1;
        if (pre[mid] <= i) li = mid;
        else hi_l = mid;
      }
      e = p.amb[(n_all * li / n_lists) * kTile + (i - pre[li])];
    }
    const bool pair = i < n && e.z >= 0;
    if (pair) {
      const int u = e.x, r = p.r_unit[u];
      const int64_t pos = e.y;
      const int j2[2] = {e.z, e.w};
      const __nv_bfloat16* krow = p.K + (int64_t(u % p.UL) * p.s + pos) * kHeadDim + 4 * c8;
      const unsigned group = 0xffu << (lane & 24);
      uint2 kw[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) kw[q] = *reinterpret_cast<const uint2*>(krow + 32 * q);
      float d2[2], nn[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float* c = p.centers32 + (int64_t(u) * p.rmax + j2[k]) * kHeadDim + 4 * c8;
        nn[k] = p.cnorm[int64_t(u) * p.rmax + j2[k]];
        float a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(c + 32 * q);
          const float2 k01 = bf16x2_to_float2(kw[q].x), k23 = bf16x2_to_float2(kw[q].y);
          const float x0 = k01.x - v.x, x1 = k01.y - v.y, x2 = k23.x - v.z, x3 = k23.y - v.w;
          a[q] = fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0)));
        }
        d2[k] = (a[0] + a[2]) + (a[1] + a[3]);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 2; ++k) d2[k] += __shfl_xor_sync(group, d2[k], o);
      float bd = INFINITY, bn = 0.f;              // the fp32 best, its centre's norm and index
      int bj = INT_MAX, na = 0;                   // (and how many may be nearest)
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (d2[k] < bd || (d2[k] == bd && j2[k] < bj)) {
          bd = d2[k];
          bn = nn[k];
          bj = j2[k];
        }
      const float hi = bj < r ? bd + interval(bd, bn) : INFINITY;
#pragma unroll
      for (int k = 0; k < 2; ++k) na += !(d2[k] - interval(d2[k], nn[k]) > hi);
      int res = bj;
      if (bj < r && na > 1) {                     // fp64 decides
        double bd64 = INFINITY;
        res = INT_MAX;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const double* c = p.centers64 + (int64_t(u) * p.rmax + j2[k]) * kHeadDim + 4 * c8;
          double a[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const double4_32a v = *reinterpret_cast<const double4_32a*>(c + 32 * q);
            const float2 k01 = bf16x2_to_float2(kw[q].x), k23 = bf16x2_to_float2(kw[q].y);
            const double kx[4] = {k01.x, k01.y, k23.x, k23.y};
            double tt = (kx[0] - v.x) * (kx[0] - v.x);
            tt = fma(kx[1] - v.y, kx[1] - v.y, tt);
            tt = fma(kx[2] - v.z, kx[2] - v.z, tt);
            a[q] = fma(kx[3] - v.w, kx[3] - v.w, tt);
          }
          double dd = (a[0] + a[2]) + (a[1] + a[3]);
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) dd += __shfl_xor_sync(group, dd, o);
          if (dd < bd64 || (dd == bd64 && j2[k] < res)) {
            bd64 = dd;
            res = j2[k];
          }
        }
      }
      if (c8 == 0) settle(u, r, pos, res);
    }
    // tokens of all centres
    if (c8 == 0 && i < n && !pair) queue[atomicAdd(&queued, 1)] = make_int2(e.x, e.y);
    __syncthreads();
    const int m = queued;
    for (int t0 = 0; t0 < m; t0 += kResWarps) {
      const int mb = min(kResWarps, m - t0);
      int r_hi = 0;
      for (int t = 0; t < mb; ++t) r_hi = max(r_hi, p.r_unit[queue[t0 + t].x]);
      const bool mine = wb < mb;                        // the token this warp decides
      const int2 tok = queue[t0 + (mine ? wb : 0)];
      const int r = p.r_unit[tok.x];
      const float* cnu = p.cnorm + int64_t(tok.x) * p.rmax;
      auto bound = [&](float d, int j) { return interval(d, cnu[j]); };
      auto key = [&](int2 t, float2& k01, float2& k23) {
        const uint2 kw = *reinterpret_cast<const uint2*>(p.K + (int64_t(t.x % p.UL) * p.s + t.y) * kHeadDim + 4 * lane);
        k01 = bf16x2_to_float2(kw.x);
        k23 = bf16x2_to_float2(kw.y);
      };
      const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
      float bd = INFINITY, hi = INFINITY;               // the fp32 best, the upper end of its interval
      int bj = INT_MAX, na = 0;                         // its index; centres that may be nearest
      bool over = false;                                // more of them than jl holds
      for (int kc = 0; kc < r_hi; kc += kResChunk) {
        // fp32 distances: a 4-term chain per lane, then for each eight centres a
        // transposed butterfly (9 shuffles) that leaves centre 4 b4 + 2 b3 + b2
        // (b_i: bit i of the lane) summed over all lanes -- five levels of adds,
        // as the bound assumes
        constexpr int kOct = 2;
        const int steps = (min(kResChunk, r_hi - kc) + 8 * kOct - 1) / (8 * kOct);
        for (int x = wb; x < mb * steps; x += kResWarps) {
          const int t = x % mb, k0 = x / mb * 8 * kOct;
          const int2 tk = queue[t0 + t];
          const int nc = min(kResChunk, p.r_unit[tk.x] - kc);
          if (k0 >= nc) continue;
          const float* c32 = p.centers32 + (int64_t(tk.x) * p.rmax + kc) * kHeadDim + 4 * lane;
          float2 k01, k23;
          key(tk, k01, k23);
          float4 c[kOct][8];
#pragma unroll
          for (int h = 0; h < kOct; ++h)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int k = k0 + 8 * h + q;
              c[h][q] = *reinterpret_cast<const float4*>(c32 + int64_t(k < nc ? k : k0) * kHeadDim);
            }
#pragma unroll
          for (int h = 0; h < kOct; ++h) {
            float a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const float x0 = k01.x - c[h][q].x, x1 = k01.y - c[h][q].y, x2 = k23.x - c[h][q].z, x3 = k23.y - c[h][q].w;
              a[q] = fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0)));
            }
            float bq[4], cq[2];
#pragma unroll
            for (int i2 = 0; i2 < 4; ++i2) {
              const float send = b4 ? a[i2] : a[i2 + 4];
              bq[i2] = (b4 ? a[i2 + 4] : a[i2]) + __shfl_xor_sync(0xffffffffu, send, 16);
            }
#pragma unroll
            for (int i2 = 0; i2 < 2; ++i2) {
              const float send = b3 ? bq[i2] : bq[i2 + 2];
              cq[i2] = (b3 ? bq[i2 + 2] : bq[i2]) + __shfl_xor_sync(0xffffffffu, send, 8);
            }
            float dq = (b2 ? cq[1] : cq[0]) + __shfl_xor_sync(0xffffffffu, b2 ? cq[0] : cq[1], 4);
            dq += __shfl_xor_sync(0xffffffffu, dq, 2);
            dq += __shfl_xor_sync(0xffffffffu, dq, 1);
            const int v = k0 + 8 * h + 4 * b4 + 2 * b3 + b2;
            if ((lane & 3) == 0 && v < nc) dsm[t][v] = dq;
          }
        }
        __syncthreads();
        const int nc = mine ? min(kResChunk, r - kc) : 0;
        // the fp32 best (distance, index)
        for (int k = lane; k < nc; k += 32) {
          const float d = dl[k];
          const int j = kc + k;
          if (d < bd || (d == bd && j < bj)) {
            bd = d;
            bj = j;
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float od = __shfl_xor_sync(0xffffffffu, bd, o);
          const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
          if (od < bd || (od == bd && oj < bj)) {
            bd = od;
            bj = oj;
          }
        }
        // the centres of the chunk whose interval reaches the best's so far
        if (bj < r) hi = bd + bound(bd, bj);
        for (int k0 = 0; k0 < nc; k0 += 32) {
          const int k = k0 + lane;
          bool m = false;
          if (k < nc) {
            const float d = dl[k];
            m = !(d - bound(d, kc + k) > hi);
          }
          const unsigned bal = __ballot_sync(0xffffffffu, m);
          if (na + __popc(bal) > kResChunk) over = true;
          else if (m) jl[na + __popc(bal & ((1u << lane) - 1u))] = kc + k;
          if (!over) na += __popc(bal);
        }
        __syncthreads();                                // dsm is refilled
      }
      int res = bj;
      if (mine && bj < r && (na > 1 || over)) {       // fp64 decides among them
        float2 k01, k23;
        key(tok, k01, k23);
        const double kx[4] = {k01.x, k01.y, k23.x, k23.y};
        const double* c64 = p.centers64 + int64_t(tok.x) * p.rmax * kHeadDim + 4 * lane;
        double bd64 = INFINITY;
        int bj64 = INT_MAX;
        const int nq = over ? r : na;
        for (int k0 = 0; k0 < nq; k0 += 4) {
          int jq[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) jq[q] = k0 + q < nq ? (over ? k0 + q : jl[k0 + q]) : -1;
          double a[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const double4_32a c =
                *reinterpret_cast<const double4_32a*>(c64 + int64_t(jq[q] < 0 ? 0 : jq[q]) * kHeadDim);
            double tt = (kx[0] - c.x) * (kx[0] - c.x);
            tt = fma(kx[1] - c.y, kx[1] - c.y, tt);
            tt = fma(kx[2] - c.z, kx[2] - c.z, tt);
            a[q] = fma(kx[3] - c.w, kx[3] - c.w, tt);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < 4; ++q) a[q] += __shfl_xor_sync(0xffffffffu, a[q], o);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const double dd = __shfl_sync(0xffffffffu, a[q], 0);
            if (jq[q] >= 0 && (dd < bd64 || (dd == bd64 && jq[q] < bj64))) {
              bd64 = dd;
              bj64 = jq[q];
            }
          }
        }
        res = bj64;
      }
      if (mine && lane == 0) settle(tok.x, r, tok.y, res);
    }
    __syncthreads();
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
  }
}

}  // namespace build
}  // namespace reskv
