// Compensated decode attention on CUDA cores for fp32 caches (bf16 caches use decode_tc.cu).
//
//   out[b][h] = sum_i softmax_i(q_h . k_i / sqrt(d) + bias_i) v_i      (Alg. 1 decode,
//                                                                     Sec. 3.6 compensation)
// Split-K flash decoding: CTA (split s, KV head kv, sequence b) streams a contiguous slice of
// the compressed rows once for all G query heads of the group, keeping a running max / sum
// per head in the base-2 domain (the bias is folded into the logit before the max).  Each CTA
// leaves (max, sum, unnormalised output) in the workspace; the last CTA of a (b, kv) to
// arrive (one atomic add, no waiting) folds the splits in split order, so the result does
// not depend on scheduling.  With k_new / v_new the new row joins the softmax with bias 0 and
// is then written at row lengths[b]; the last (b, kv) of a sequence bumps lengths[b].
#include <algorithm>

#include "decode_common.cuh"
#include "selkv_internal.cuh"

namespace selkv {
namespace {

// A warp takes kLoads loads of K and as many of V at a time, all in flight together: a lane holds
// four elements of a row, so D / 4 lanes share a row and a step covers kLoads * 128 / D keys.
// Small caches are bound by latency, a token of one sequence of 256 rows by its whole chain: with
// a row per lane (its elements loaded eight at a time, values row by row) that launch took 27 us, now
// 11 (both from a cold L2).
constexpr int kLoads = 8;
// Warps of a CTA (the fold's scratch stays within 48 KB of static shared memory).
constexpr int warps_of(int GM) { return GM <= 8 ? 8 : 4; }

// Sums of x[i] over the D / 4 lanes of a row, spread over them: every level keeps half of the
// values and adds the partner's, so a lane ends with the sum of one i, given by its lane bits.
template <int LPR>
__device__ __forceinline__ float spread_sum(const float (&x)[kLoads], int lane) {
  float q[kLoads];
#pragma unroll
  for (int i = 0; i < kLoads; ++i) q[i] = x[i];
#pragma unroll
  for (int o = LPR / 2, keep = kLoads; o > 0; o >>= 1) {
    const bool up = lane & o;
    if (keep > 1) {
      keep >>= 1;
#pragma unroll
      for (int i = 0; i < keep; ++i) {
        const float mine = up ? q[keep + i] : q[i], other = up ? q[i] : q[keep + i];
        q[i] = mine + __shfl_xor_sync(0xffffffffu, other, o);
      }
    } else {
      q[0] += __shfl_xor_sync(0xffffffffu, q[0], o);
    }
  }
  return q[0];
}

template <typename T, int D, int GM>
__global__ __launch_bounds__(warps_of(GM) * 32) void decode_simt_kernel(DecodeArgs a) {
  constexpr int kWarps = warps_of(GM);
  constexpr int LPR = D / 4, RPI = 32 / LPR;  // lanes per row, rows per load
  constexpr int kKeys = kLoads * RPI;         // keys of a warp's step
  constexpr int kLow = LPR / kLoads;          // lanes that end with the same sum
  static_assert(kLow >= 1, "a row's lanes hold every sum");
  __shared__ __align__(16) float qs[GM][D];
  __shared__ float wm[kWarps][GM], wl[kWarps][GM];
  __shared__ __align__(16) float wo[kWarps][GM][D];
  __shared__ bool s_last;
  const int s = blockIdx.x, kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = a.G, S = a.splits;
  const size_t bk = (size_t)b * a.Hkv + kv;

  int L = a.lengths[b];
  for (int i = tid; i < G * D; i += blockDim.x) {
    const int g = i / D, d = i % D;
    qs[g][d] = load1(static_cast<const T*>(a.q) + ((size_t)b * a.Hq + kv * G + g) * D + d) * a.scale_log2;
  }
  if (L < 0 || L > a.m_cap) {
    if (tid == 0 && s == 0 && kv == 0) raise_flag(a.flags, SELKV_DEVERR_LENGTH);
    L = L < 0 ? 0 : a.m_cap;
  }
  bool app = a.k_new != nullptr;
  if (app && L + 1 > a.m_cap) {
    if (tid == 0 && s == 0 && kv == 0) raise_flag(a.flags, SELKV_DEVERR_CAPACITY);
    app = false;
  }
  const int total = L + (app ? 1 : 0);
  const int chunk = ((total + S - 1) / S + 31) / 32 * 32;
  const int lo = s * chunk, hi = min(total, lo + chunk);
  __syncthreads();

  const T* Kb = static_cast<const T*>(a.Kc) + bk * a.m_cap * D;
  const T* Vb = static_cast<const T*>(a.Vc) + bk * a.m_cap * D;
  const T* kn = app ? static_cast<const T*>(a.k_new) + bk * D : nullptr;
  const T* vnw = app ? static_cast<const T*>(a.v_new) + bk * D : nullptr;
  const float* bias = a.bias != nullptr ? a.bias + bk * a.m_cap : nullptr;

  const int sub = lane / LPR, e0 = (lane % LPR) * 4;
  // the key of a step whose logit this lane ends with: load `mine` of its row group
  const int mine = (lane % LPR) / kLow;
  float m[GM], l[GM], o[GM][4];
#pragma unroll
  for (int g = 0; g < GM; ++g) {
    m[g] = -INFINITY;
    l[g] = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) o[g][e] = 0.f;
  }
  for (int t0 = lo + warp * kKeys; t0 < hi; t0 += kWarps * kKeys) {
    float k[kLoads][4], v[kLoads][4];
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int key = t0 + i * RPI + sub;
      if (key < hi) {
        load4((key < L ? Kb + (size_t)key * D : kn) + e0, k[i]);
        load4((key < L ? Vb + (size_t)key * D : vnw) + e0, v[i]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) k[i][e] = v[i][e] = 0.f;
      }
    }
    const int key = t0 + mine * RPI + sub;
    const bool valid = key < hi;
    const float bv = (key < min(hi, L) && bias != nullptr) ? bias[key] * kLog2e : 0.f;
#pragma unroll
    for (int g = 0; g < GM; ++g) {
      if (g >= G) break;
      const float4 q = *reinterpret_cast<const float4*>(&qs[g][e0]);
      float part[kLoads];
#pragma unroll
      for (int i = 0; i < kLoads; ++i)
        part[i] = fmaf(k[i][3], q.w, fmaf(k[i][2], q.z, fmaf(k[i][1], q.y, k[i][0] * q.x)));
      const float dot = spread_sum<LPR>(part, lane);
      const float x = valid ? dot + bv : -INFINITY;
      float mx = x;
#pragma unroll
      for (int d = kLow; d < 32; d <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
      const float mn = fmaxf(m[g], mx);
      const float mref = mn == -INFINITY ? 0.f : mn;  // (so far every key has weight 0)
      const float corr = exp2f(m[g] - mref);
      const float p = exp2f(x - mref);
      float ps = p;
#pragma unroll
      for (int d = kLow; d < 32; d <<= 1) ps += __shfl_xor_sync(0xffffffffu, ps, d);
      l[g] = l[g] * corr + ps;
#pragma unroll
      for (int e = 0; e < 4; ++e) o[g][e] *= corr;
      m[g] = mn;
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        const float pi = __shfl_sync(0xffffffffu, p, sub * LPR + i * kLow);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[g][e] = fmaf(pi, v[i][e], o[g][e]);
      }
    }
  }
  // fold the warps
#pragma unroll
  for (int g = 0; g < GM; ++g) {
    if (g >= G) break;
    if (lane == 0) {
      wm[warp][g] = m[g];
      wl[warp][g] = l[g];
    }
    // the row groups of a warp share its max and sum: their outputs are added
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int d = LPR; d < 32; d <<= 1) o[g][e] += __shfl_xor_sync(0xffffffffu, o[g][e], d);
    if (sub == 0) *reinterpret_cast<float4*>(&wo[warp][g][e0]) = make_float4(o[g][0], o[g][1], o[g][2], o[g][3]);
  }
  __syncthreads();
  write_split_partial<kWarps>(a, b, kv, s, &wo[0][0][0], &wm[0][0], &wl[0][0], GM, D, false);
  if (!arrive_last(a, bk, &s_last)) return;
  combine_splits<T>(a, b, kv, &wo[0][0][0]);
  if (app) write_append_row<T>(a, bk, L, threadIdx.x, blockDim.x);
  finish_lengths(a, b, bk, L, app);
}

template <typename T, int D>
cudaError_t launch_t(const DecodeArgs& a, cudaStream_t st) {
  const dim3 grid(a.splits, a.Hkv, a.B);
  if (a.G <= 1) decode_simt_kernel<T, D, 1><<<grid, warps_of(1) * 32, 0, st>>>(a);
  else if (a.G <= 2) decode_simt_kernel<T, D, 2><<<grid, warps_of(2) * 32, 0, st>>>(a);
  else if (a.G <= 4) decode_simt_kernel<T, D, 4><<<grid, warps_of(4) * 32, 0, st>>>(a);
  else if (a.G <= 8) decode_simt_kernel<T, D, 8><<<grid, warps_of(8) * 32, 0, st>>>(a);
  else decode_simt_kernel<T, D, 16><<<grid, warps_of(16) * 32, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

#ifndef SELKV_DEC_CTAS_PER_SM
#define SELKV_DEC_CTAS_PER_SM 1  // decode CTAs planned per SM when splitting the rows
#endif
#ifndef SELKV_DEC_FILL_ROWS
#define SELKV_DEC_FILL_ROWS 256  // a CTA's fixed cost in the split model, in rows streamed
#endif
#ifndef SELKV_DEC_BACKFILL_WAVES
#define SELKV_DEC_BACKFILL_WAVES 3  // one split over at least this many waves of units ...
#endif
#ifndef SELKV_DEC_BACKFILL_MAX_ROWS
#define SELKV_DEC_BACKFILL_MAX_ROWS 8192  // ... of at most this many rows: fractional waves
#endif
#ifndef SELKV_DEC_MAX_SPLITS
#define SELKV_DEC_MAX_SPLITS 64  // most splits of one (sequence, KV head)
#endif

// Split count of each (sequence, KV head).  The B * Hkv * S CTAs run in waves of
// CTAS_PER_SM * num_sms; a wave lasts about as long as streaming one CTA's rows plus a fixed
// fill-and-fold cost worth kFillRows rows.  S minimises waves * (rows per CTA + kFillRows) over
// the capacity m_cap, fewest splits on ties.  With `unit_walk` (the tensor-core decode), one
// split over more units than slots with at most SELKV_DEC_UNITS_MAX_ROWS rows runs as
// persistent CTAs that pay the fixed cost once: waves * rows + kFillRows (the walk priced as the one CTA
// per SM on 128-row tiles that it was; with 64-row tiles and two it is faster than that).  There too, one split
// over at least BACKFILL_WAVES waves of units of at most BACKFILL_MAX_ROWS rows counts its waves as
// units / slots: the block scheduler starts each unit as a slot frees, so ragged units pack
// (batch 64 x 8k at 50%: 151.0 -> 144.0 us per launch, 64 x 32k at 10%: 129.6 -> 120.7; with
// longer units the last ones started leave a tail: 64 x 32k at 50% 490 -> 496, 64 x 128k at
// 25% 924 -> 972, so those keep their splits).  (Serving sweep, batch 8 x 32k at 50%: 256
// rows of fixed cost pick more splits than 512 did, 85.7 -> 71.0 us per launch; batch 4 x 8k:
// 4 splits either way.)
int decode_splits(int B, int Hkv, int m_cap, int num_sms, bool unit_walk) {
  constexpr long kFillRows = SELKV_DEC_FILL_ROWS;
  const long units = (long)B * Hkv;
  const long slots = std::max(1L, (long)SELKV_DEC_CTAS_PER_SM * num_sms);
  const int smax = std::max(1, std::min(SELKV_DEC_MAX_SPLITS, (m_cap + 63) / 64));
  int best = 1;
  long best_cost = -1;
  for (int S = 1; S <= smax; ++S) {
    // costs in units of rows x slots, so that fractional waves stay integral
    const long waves = (units * S + slots - 1) / slots * slots;
    const long rows = ((long)(m_cap + S - 1) / S + 63) / 64 * 64;
    const bool walk = unit_walk && S == 1 && units > slots && m_cap <= SELKV_DEC_UNITS_MAX_ROWS;
    const bool backfill = unit_walk && S == 1 && !walk && units >= (long)SELKV_DEC_BACKFILL_WAVES * slots &&
                          m_cap <= SELKV_DEC_BACKFILL_MAX_ROWS;
    const long cost = walk ? waves * rows + kFillRows * slots
                           : (backfill ? units : waves) * (rows + kFillRows);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = S;
    }
  }
  return best;
}

cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t st) {
  if (a.dtype == SELKV_BF16) return launch_decode_tc(a, st);
  return a.D == 128 ? launch_t<float, 128>(a, st) : launch_t<float, 64>(a, st);
}

}  // namespace selkv
