// Decode-time growth of the cache (Sec. 3.1: each decode step appends the new
// token's key and value): one exact K row and V row per (batch, KV head) unit
// goes after the unit's main and residual slots and counts as a main-cache
// token from then on.
//
// The A slots after the residual entries hold the unit's appended tokens as a
// ring: token t (counted from the first append) sits at ring index t mod A.
// While fewer than A tokens were appended the new one takes the next free
// slot.  Once the ring is full the oldest token (index n_total mod A) leaves
// the exact window before the new token takes its slot; the append policy
// decides what becomes of it:
//   RESKV_APPEND_RING_DROP: it leaves the cache;
//   RESKV_APPEND_RING_FOLD: it becomes a member of its nearest residual entry
//     (Eq. residual_partition's nearest-centre rule on the stored keys, ties
//     to the lower entry), whose stored means and count are updated as a
//     running mean (Eq. summary): k_bar <- (c k_bar + k) / (c + 1) in fp64,
//     rounded to bf16, likewise v_bar, c <- c + 1, log-count beta log(c + 1).
//     A unit without residual entries drops the token.  This is the residual
//     refresh during generation that the paper leaves to future work (App. E).
//
// The nearest entry is decided exactly, in two steps.  First every entry's
// distance is taken in fp32 as sum_i (k_i - k_bar_ji)^2, which has no
// cancellation: its relative error is at most 16 u (u = 2^-24: a rounded
// difference, its square, a chain of 4 terms, 5 butterfly levels), plus an
// absolute part from underflow.  An entry whose interval does not reach the
// best one's cannot be nearest, so usually a single entry is left.  Where
// several are, they are compared exactly: with every bf16 value written as
// M 2^e (integer M < 2^8), ||k - k_bar_j||^2 - ||k||^2 = sum_i (k_bar_ji^2 -
// 2 k_i k_bar_ji) is a signed sum of terms m 2^t with integer m < 2^17, one
// lane per entry; within the exponent window of the rows involved the terms
// are integers of a common scale that a signed 128-bit sum holds, and rows
// that span more than that window are decided by one lane with a 576-bit
// accumulator of 32-bit digits.
//
// What bounds it: latency.  A unit reads at most a few hundred 256-byte entry
// rows (51 KB at 204 entries) and writes four rows, so the time is a chain of
// dependent loads: the counts, the rows, the chosen entry.  One CTA of 8 warps
// per unit keeps 64 rows in flight; the launch is a programmatic dependent
// launch, and everything up to the new token's rows is read before the wait
// for the previous kernel, which is a decode that only reads the cache.  (On the
// SMs the decode leaves free: a CTA of 98 registers x 256 threads does not fit
// beside one of the cluster decode's 200 x 256.)
// Measured on 64 units a layer with 0..204 entries (32K, b = 1024, B = 8), an
// append and a decode per layer: 17.3 us a layer, of which the decode alone
// takes 7.9; 244 us before, when one warp per unit took the 128-bit sums over
// every entry and was bound by that integer chain of 128 dims.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "device_utils.cuh"
#include "internal.h"

namespace reskv {
namespace {

using i128 = __int128;

struct AppendArgs {
  const __nv_bfloat16* K_new;   // [n, d]
  const __nv_bfloat16* V_new;
  __nv_bfloat16* kslots;
  __nv_bfloat16* vslots;
  float* logc;
  int32_t* slot_pos;
  int32_t* counts;
  const int32_t* n_main;
  const int32_t* n_res;
  int32_t* n_app;               // appended tokens in the cache, min(n_total, A)
  int32_t* n_total;             // tokens appended since construction
  const int32_t* offsets;       // [U+1] unit starts, or NULL (uniform stride)
  int64_t unit0;
  int32_t stride;
  int32_t capacity;             // A
  int32_t policy;               // RESKV_APPEND_*
  float beta;
  int64_t seq_len;
  uint32_t* status;
};

// A bf16 value as sign, integer M (< 2^8) and exponent e: value = +-M 2^e.
struct Bf {
  uint32_t m;
  int e;
  uint32_t neg;
};

__device__ __forceinline__ Bf bf_split(uint16_t b) {
  const uint32_t ef = (b >> 7) & 0xffu, mf = b & 0x7fu;
  return Bf{ef ? 128u + mf : mf, int(ef ? ef : 1u) - 134, uint32_t(b >> 15)};
}

__device__ __forceinline__ bool bf_finite(uint16_t b) { return ((b >> 7) & 0xffu) != 0xffu; }

// ---- the 576-bit accumulator of the wide case (one thread) ----------------
// Digit q holds bits 32q..32q+31 of the sum scaled by 2^266 (t >= -266).
constexpr int kDigits = 18;

__device__ void wide_add(int64_t* dig, uint32_t m, int t, bool negative) {
  const int q = t + 266;
  const uint64_t v = uint64_t(m) << (q & 31);
  const int64_t lo = int64_t(v & 0xffffffffu), hi = int64_t(v >> 32);
  dig[q >> 5] += negative ? -lo : lo;
  dig[(q >> 5) + 1] += negative ? -hi : hi;
}

// Carries into the upper digits; afterwards every digit but the top one is in
// [0, 2^32) and the top digit carries the sign.
__device__ void wide_normalise(int64_t* dig) {
  for (int q = 0; q < kDigits - 1; ++q) {
    const int64_t carry = dig[q] >> 32;          // arithmetic shift: floor division
    dig[q] -= carry * (int64_t(1) << 32);
    dig[q + 1] += carry;
  }
}

// -1, 0, 1 as a < b, a == b, a > b (both normalised).
__device__ int wide_cmp(const int64_t* a, const int64_t* b) {
  for (int q = kDigits - 1; q >= 0; --q)
    if (a[q] != b[q]) return a[q] < b[q] ? -1 : 1;
  return 0;
}

// The entry of list[0 .. n) (NULL: 0 .. n - 1) nearest to key k (rows kb),
// exactly, ties to the lower entry, by one thread.
__device__ int nearest_wide(const uint16_t* k, const uint16_t* kb, const int* list, int n) {
  int64_t best[kDigits], cur[kDigits];
  int bj = INT_MAX;
  for (int x = 0; x < n; ++x) {
    const int j = list ? list[x] : x;
    for (int q = 0; q < kDigits; ++q) cur[q] = 0;
    for (int i = 0; i < kHeadDim; ++i) {
      const Bf b = bf_split(kb[size_t(j) * kHeadDim + i]);
      if (!b.m) continue;
      wide_add(cur, b.m * b.m, 2 * b.e, false);
      const Bf a = bf_split(k[i]);
      if (a.m) wide_add(cur, 2u * a.m * b.m, a.e + b.e, a.neg == b.neg);
    }
    wide_normalise(cur);
    const int c = x == 0 ? -1 : wide_cmp(cur, best);
    if (c < 0 || (c == 0 && j < bj)) {
      bj = j;
      for (int q = 0; q < kDigits; ++q) best[q] = cur[q];
    }
  }
  return bj;
}

// The same by one warp: 128-bit sums, one entry per lane, where the rows'
// exponents allow.  Every value must be finite.
__device__ __noinline__ int nearest_exact(const uint16_t* k, const uint16_t* kb, const int* list, int n) {
  const int lane = threadIdx.x & 31;
  // the exponent window: the largest exponent of any value involved
  int emax = INT_MIN;
  for (int x = lane; x < (n + 1) * kHeadDim; x += 32) {
    const int row = x / kHeadDim - 1, d = x % kHeadDim;
    const uint16_t bits = row < 0 ? k[d] : kb[size_t(list ? list[row] : row) * kHeadDim + d];
    const Bf b = bf_split(bits);
    if (b.m) emax = max(emax, b.e);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  // terms m 2^t (m < 2^17) as integers of scale 2^base; every |term| <
  // 2^(2 emax + 17) and 2 * 128 terms sum below 2^(2 emax + 25) < 2^(base + 127)
  const int base = emax == INT_MIN ? 0 : 2 * emax - 102;
  bool wide = false;
  i128 dbest = 0;
  int jbest = INT_MAX;
  for (int x = lane; x < n; x += 32) {
    const int j = list ? list[x] : x;
    i128 acc = 0;
    for (int d = 0; d < kHeadDim; ++d) {
      const Bf b = bf_split(kb[size_t(j) * kHeadDim + d]);
      if (!b.m) continue;
      const int t2 = 2 * b.e - base;
      if (t2 < 0) wide = true;
      else acc += i128(b.m * b.m) << t2;
      const Bf c = bf_split(k[d]);
      if (!c.m) continue;
      const int t1 = c.e + b.e - base;
      if (t1 < 0) {
        wide = true;
        continue;
      }
      const i128 pr = i128(2u * c.m * b.m) << t1;
      acc += c.neg == b.neg ? -pr : pr;
    }
    if (jbest == INT_MAX || acc < dbest || (acc == dbest && j < jbest)) {
      dbest = acc;
      jbest = j;
    }
  }
  if (__any_sync(0xffffffffu, wide)) {
    const int j = lane == 0 ? nearest_wide(k, kb, list, n) : 0;
    return __shfl_sync(0xffffffffu, j, 0);
  }
  // warp argmin, ties to the lower entry (lanes without an entry hold INT_MAX)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t hi = __shfl_xor_sync(0xffffffffu, uint64_t((unsigned __int128)(dbest) >> 64), o);
    const uint64_t lo = __shfl_xor_sync(0xffffffffu, uint64_t(dbest), o);
    const int jo = __shfl_xor_sync(0xffffffffu, jbest, o);
    const i128 d_o = i128((unsigned __int128)(hi) << 64 | lo);
    if (jo != INT_MAX && (jbest == INT_MAX || d_o < dbest || (d_o == dbest && jo < jbest))) {
      dbest = d_o;
      jbest = jo;
    }
  }
  return jbest;
}

constexpr int kAppWarps = 8;
constexpr int kAppThreads = kAppWarps * 32;
constexpr int kAppChunk = 1024;         // entries whose fp32 distances are held at once
constexpr int kAppCand = 64;            // entries left for the exact comparison, at most

// Half-width of the interval around an fp32 distance that holds the exact one.
__device__ __forceinline__ float dist_bound(float d) { return 1.2e-6f * d + 1e-40f; }

// The residual entry of [0, nr) (rows kb) nearest to key k, exactly, ties to
// the lower entry; -1 if a value of k or of an entry is not finite.  Every
// thread of the CTA calls it and gets the answer.
__device__ int nearest_entry(const uint16_t* k, const uint16_t* kb, int nr) {
  __shared__ float dist[kAppChunk];
  __shared__ float wmin[kAppWarps];
  __shared__ int cand[kAppCand], ncand, odd, answer;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint2 kw = *reinterpret_cast<const uint2*>(k + 4 * lane);
  const float2 k01 = bf16x2_to_float2(kw.x), k23 = bf16x2_to_float2(kw.y);
  const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
  if (threadIdx.x == 0) ncand = odd = 0;
  __syncthreads();                      // (any warp may raise odd)
  float hi = INFINITY;                  // least upper end of an interval so far
  for (int c0 = 0; c0 < nr; c0 += kAppChunk) {
    const int nc = min(kAppChunk, nr - c0);
    float mn = INFINITY;
    // eight entries at a time per warp: a 4-term chain per lane, then a
    // transposed butterfly that leaves entry 4 b4 + 2 b3 + b2 summed over the
    // lanes (five levels)
    for (int j0 = 8 * w; j0 < nc; j0 += 8 * kAppWarps) {
      uint2 e[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        e[q] = *reinterpret_cast<const uint2*>(kb + size_t(c0 + min(j0 + q, nc - 1)) * kHeadDim + 4 * lane);
      float a[8], bq[4], cq[2];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float2 e01 = bf16x2_to_float2(e[q].x), e23 = bf16x2_to_float2(e[q].y);
        const float x0 = k01.x - e01.x, x1 = k01.y - e01.y, x2 = k23.x - e23.x, x3 = k23.y - e23.y;
        a[q] = fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0)));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        bq[i] = (b4 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, b4 ? a[i] : a[i + 4], 16);
#pragma unroll
      for (int i = 0; i < 2; ++i)
        cq[i] = (b3 ? bq[i + 2] : bq[i]) + __shfl_xor_sync(0xffffffffu, b3 ? bq[i] : bq[i + 2], 8);
      float dq = (b2 ? cq[1] : cq[0]) + __shfl_xor_sync(0xffffffffu, b2 ? cq[0] : cq[1], 4);
      dq += __shfl_xor_sync(0xffffffffu, dq, 2);
      dq += __shfl_xor_sync(0xffffffffu, dq, 1);
      const int v = j0 + 4 * b4 + 2 * b3 + b2;
      if ((lane & 3) == 0 && v < nc) {
        dist[v] = dq;
        if (!(dq < INFINITY)) odd = 1;   // a value that is not finite, or an overflow
        mn = fminf(mn, dq);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    if (lane == 0) wmin[w] = mn;
    __syncthreads();
    mn = wmin[0];
#pragma unroll
    for (int i = 1; i < kAppWarps; ++i) mn = fminf(mn, wmin[i]);
    hi = fminf(hi, mn + dist_bound(mn));
    // entries of this chunk that may be nearest (those of earlier chunks stay)
    for (int j = threadIdx.x; j < nc; j += kAppThreads)
      if (!(dist[j] - dist_bound(dist[j]) > hi)) {
        const int x = atomicAdd(&ncand, 1);
        if (x < kAppCand) cand[x] = c0 + j;
      }
    __syncthreads();
  }
  if (ncand == 1 && odd == 0) return cand[0];
  // several are left: compared exactly, or every entry where the list is
  // too short or a distance is not a finite number
  bool finite = true;
  if (odd != 0)
    for (int x = threadIdx.x; x < (nr + 1) * kHeadDim; x += kAppThreads)
      finite &= bf_finite(x < kHeadDim ? k[x] : kb[x - kHeadDim]);
  if (!__syncthreads_and(finite)) return -1;
  if (w == 0) {
    const bool all = odd != 0 || ncand > kAppCand;
    const int j = nearest_exact(k, kb, all ? nullptr : cand, all ? nr : ncand);
    if (lane == 0) answer = j;
  }
  __syncthreads();
  return answer;
}

// One CTA per unit of the call; thread t < 128 holds dim t of the keys, thread
// 128 + t dim t of the values.
__global__ void __launch_bounds__(kAppThreads) k_append(AppendArgs a) {
  const int64_t i = blockIdx.x, u = a.unit0 + i;
  const int tid = threadIdx.x;
  // Before the wait: the counts and the cache, which only appends write, and
  // no append is running: it lets no later kernel start before its end.
  const int total = a.n_total[u];
  const int64_t ubase = a.offsets ? int64_t(a.offsets[u]) : u * a.stride;
  const int nm = a.n_main[u], nr = a.n_res[u];
  const int64_t ring0 = ubase + nm + nr;            // first appended slot
  const bool full = total >= a.capacity;
  const bool refuse = full && (a.policy == RESKV_APPEND_FAIL || a.capacity == 0);   // the host checks first
  const int64_t row = ring0 + (a.capacity > 0 ? total % a.capacity : 0);
  __nv_bfloat16* const slots = tid < kHeadDim ? a.kslots : a.vslots;
  const int d = tid & (kHeadDim - 1);
  int best = -1, c = 0;
  bool dropped = false;
  int64_t erow = 0;
  __nv_bfloat16 mean{};
  if (!refuse && full && a.policy == RESKV_APPEND_RING_FOLD && nr > 0) {
    // the oldest appended token, k and v of slot `row`, joins its nearest entry
    best = nearest_entry(reinterpret_cast<const uint16_t*>(a.kslots + row * kHeadDim),
                         reinterpret_cast<const uint16_t*>(a.kslots + (ubase + nm) * kHeadDim), nr);
    dropped = best < 0;                              // distances undefined: dropped instead
    if (best >= 0) {
      // running mean of the stored summary and the token, one value per thread
      erow = ubase + nm + best;
      c = a.counts[erow];
      const double cd = double(c);
      const double xo = double(__bfloat162float(slots[row * kHeadDim + d]));
      const double xe = double(__bfloat162float(slots[erow * kHeadDim + d]));
      mean = __double2bfloat16(__ddiv_rn(__dadd_rn(__dmul_rn(cd, xe), xo), cd + 1.0));
    }
  }
  // K_new and V_new, and every write, only after the previous kernel on the
  // stream (which may read the slots written here) has completed
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();                                   // every thread has read what is overwritten
  if (refuse) {
    if (tid == 0) report_status(a.status, kStatusBadIndex);
    return;
  }
  if (best >= 0) {
    slots[erow * kHeadDim + d] = mean;
    if (tid == 0) {
      a.counts[erow] = c + 1;
      a.logc[erow] = a.beta * logf(float(c + 1));
    }
  }
  // the new token into slot `row`
  if (tid < 16) {
    reinterpret_cast<uint4*>(a.kslots + row * kHeadDim)[tid] =
        reinterpret_cast<const uint4*>(a.K_new + i * kHeadDim)[tid];
  } else if (tid < 32) {
    reinterpret_cast<uint4*>(a.vslots + row * kHeadDim)[tid - 16] =
        reinterpret_cast<const uint4*>(a.V_new + i * kHeadDim)[tid - 16];
  } else if (tid == 32) {
    a.slot_pos[row] = int32_t(a.seq_len + total);    // position of the token in the sequence
    a.counts[row] = 0;
    a.logc[row] = 0.f;
    a.n_total[u] = total + 1;
    a.n_app[u] = total + 1 < a.capacity ? total + 1 : a.capacity;
    if (dropped) report_status(a.status, kStatusBadIndex);
  }
  // The rows are visible device-wide before this grid completes: decode
  // kernels launched after it read the cache before their own grid
  // dependency wait.
  __threadfence();
}

}  // namespace

cudaError_t launch_append(reskv_cache* c, int64_t unit0, int64_t n, const __nv_bfloat16* K_new,
                          const __nv_bfloat16* V_new, cudaStream_t stream) {
  AppendArgs a{K_new, V_new, c->kslots, c->vslots, c->logc, c->slot_pos, c->counts,
               c->n_main, c->n_res, c->n_app, c->n_total, c->ragged ? c->offsets : nullptr,
               unit0, c->stride, c->append_capacity, c->cfg.append_policy, c->cfg.beta,
               c->cfg.seq_len, c->status};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(n), 1, 1);
  cfg.blockDim = dim3(kAppThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see griddepcontrol.wait
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t err = cudaLaunchKernelEx(&cfg, k_append, a);
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace reskv
