// Pooling and the shared-set selection of SelKV, a thread-block cluster per selection.
//
//   c^_j  = (1/K) sum_{|t| <= K/2, 0 <= j+t < n_b - m_r} a_{j+t} ||v_{j+t}||   (Eq. 1, Sec. 3.2)
//   T_kv  = top-m_s of c^ over the candidates [0, n_b - m_r)                    (Eq. 2)
//   U     = union over KV heads; if |U| > m_s, keep the top-m_s of U by the score summed
//           over KV heads (the order of the mean of Sec. 3.3); then the recent window.
// Every top-k orders by value descending, then position ascending, and is an exact radix
// select on the fp32 bit patterns (scores are >= 0, so unsigned order = numeric order), done
// in three digit passes (11, 10, 10 bits).  A selection selects j iff bits(key_j) > T or
// (bits(key_j) == T and j <= jcut).
//
// Two kernels: topk_kernel pools and selects per (sequence, KV head), and in the per-head mode
// compacts that head's set; trim_kernel (shared mode) forms the union, trims it and compacts.
// A cluster of 1-16 CTAs owns one selection: each CTA keeps the keys of a contiguous span of
// positions in shared memory and counts their digits there; after one cluster barrier every CTA
// finds the digit for itself from the others' counts, read through distributed shared memory
// (first the sums of 16 slices of the bins, then the bins of one slice).  A grid-wide pass cost a
// launch, a histogram in L2, an arrival and a last CTA working alone: the selection was eight such
// kernels and a memset, 75 us for one layer of 8 x 100k and 61 us at 8 x 16k; now 43 and 26 us (each
// kernel alone, from a cold start).
// What bounds it is latency: a CTA walks its positions with a few loads in flight a warp, then
// three passes of barriers and remote reads.  Nothing waits outside the cluster.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "cluster_fit.h"
#include "ptx.cuh"
#include "selkv_internal.cuh"

namespace selkv {
namespace {

constexpr int kMaxCluster = 16;
constexpr int kMaxSpan = 24576;  // positions of a CTA whose keys are held in shared memory (96 KB)
constexpr uint32_t kNoKey = 0xFFFFFFFFu;  // not a candidate (no score has this bit pattern)

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier over the cluster's threads; orders shared-memory accesses of its CTAs.  One CTA: a
// CTA barrier.
__device__ __forceinline__ void cluster_sync(int cs) {
  if (cs == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}
// The two halves of a first barrier of the cluster: shared memory of another CTA may be touched only
// once that CTA runs.  The work between the halves hides the wait.
__device__ __forceinline__ void cluster_started_arrive(int cs) {
  if (cs > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_started_wait(int cs) {
  if (cs > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t ld_peer(const uint32_t* p, int rank) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer(uint32_t* p, int rank, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(p, rank)), "r"(v) : "memory");
}

// Digit passes over bits 30-20, 19-10 and 9-0 (a score's sign bit is 0), a histogram each, and
// the sums of its kSlices slices of bins.
constexpr int kSlices = 16;
__host__ __device__ constexpr int pass_bins(int pass) { return pass == 0 ? 2048 : 1024; }
__host__ __device__ constexpr int pass_shift(int pass) { return pass == 0 ? 20 : pass == 1 ? 10 : 0; }
__host__ __device__ constexpr int pass_off(int pass) { return pass == 0 ? 0 : 1024 + 1024 * pass; }

template <int NT>  // threads per CTA
struct Shared {
  uint32_t hist[4096];           // the three passes' digit counts of this CTA's keys
  uint32_t coarse[3][kSlices];   // and their sums over each slice of the bins
  uint32_t part[NT];             // the chosen slice's bins, summed over some of the cluster's CTAs
  uint32_t cnt[2][kMaxCluster];  // per-CTA counts of a position-ordered rank, two uses in turn
  uint32_t wsum[NT / 32];
  uint32_t slice, above, digit, before, in_digit;
  int jcut;
};

// One selection's geometry as a CTA sees it: its span of positions, kept as keys in shared
// memory (or in `far`, in global memory, where a span is too long), a contiguous part of it per warp.
struct Span {
  int cs, rank;   // cluster size, this CTA's rank
  int base, len;  // positions [base, base + len); len is a multiple of NT
  int wlo, wlen;  // this warp's part, relative to base
  uint32_t* keys;
};
template <int NT>
__device__ __forceinline__ Span make_span(int n, int cs, uint32_t* near_keys, uint32_t* far) {
  Span s;
  s.cs = cs;
  s.rank = cs == 1 ? 0 : (int)cluster_rank();
  s.len = ((n + cs - 1) / cs + NT - 1) / NT * NT;
  s.base = s.rank * s.len;
  s.wlen = s.len / (NT / 32);
  s.wlo = (threadIdx.x >> 5) * s.wlen;
  s.keys = near_keys != nullptr ? near_keys : far + s.base;
  return s;
}
// Ends of the warp's part that hold positions below `hi` (a warp-uniform trip count).
__device__ __forceinline__ int part_end(const Span& s, int hi) {
  return min(s.wlo + s.wlen, max(s.wlo, (hi - s.base + 31) & ~31));
}

// Exclusive sum of `v` over the CTA's warps (every lane passes its warp's value) and the total.
template <int NT>
__device__ __forceinline__ uint32_t scan_warps(Shared<NT>& sh, uint32_t v, uint32_t& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh.wsum[warp] = v;
  __syncthreads();
  constexpr int kWarps = NT / 32;
  const uint32_t x = lane < kWarps ? sh.wsum[lane] : 0u;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < kWarps; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  total = __shfl_sync(0xffffffffu, incl, kWarps - 1);
  const uint32_t excl = __shfl_sync(0xffffffffu, incl - x, warp);
  __syncthreads();
  return excl;
}
// The same over the whole cluster, in rank order.  `use` alternates between consecutive calls.
template <int NT>
__device__ __forceinline__ uint32_t scan_cluster(Shared<NT>& sh, const Span& s, int use, uint32_t v, uint32_t& total) {
  uint32_t cta;
  uint32_t excl = scan_warps(sh, v, cta);
  if (s.cs == 1) {
    total = cta;
    return excl;
  }
  if ((int)threadIdx.x < s.cs) st_peer(&sh.cnt[use][s.rank], threadIdx.x, cta);
  cluster_sync(s.cs);
  total = 0u;
  for (int r = 0; r < s.cs; ++r) {
    const uint32_t c = sh.cnt[use][r];
    if (r < s.rank) excl += c;
    total += c;
  }
  return excl;
}

// From the top, the bin that holds the krem-th entry: lane i of a warp has the counts c[0..N-1]
// of bins top - N i, top - N i - 1, ...  The lane that finds it calls found(index from the top,
// entries above the bin, entries in it).
template <int N, typename F>
__device__ __forceinline__ void find_bin(const uint32_t (&c)[N], uint32_t krem, F found) {
  const int lane = threadIdx.x & 31;
  uint32_t own = 0u;
#pragma unroll
  for (int t = 0; t < N; ++t) own += c[t];
  uint32_t incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  uint32_t cum = incl - own;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    if (cum < krem && cum + c[t] >= krem) found(lane * N + t, cum, c[t]);
    cum += c[t];
  }
}

// One digit pass: the counts of pass `PASS` in sh.hist (complete after the barrier here) give the
// digit that holds the krem-th largest; narrows prefix and krem.  `in_digit` gets its count.
// Every CTA of the cluster finds it for itself, in two rounds of reads from the others: the
// slice sums, then the bins of one slice.  A pass has its own histogram, so one cluster barrier
// a pass is enough.
template <int PASS, int NT>
__device__ __forceinline__ void pick_digit(Shared<NT>& sh, const Span& s, uint32_t& prefix, uint32_t& krem,
                                           uint32_t& in_digit) {
  constexpr int kPer = pass_bins(PASS) / kSlices;  // bins per slice: 128 or 64
  constexpr int kLaneBins = kPer / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t* hist = sh.hist + pass_off(PASS);
  __syncthreads();  // this CTA's counts are in
  if (warp < kSlices) {
    uint32_t v = 0u;
#pragma unroll
    for (int t = 0; t < kLaneBins; ++t) v += hist[warp * kPer + t * 32 + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh.coarse[PASS][warp] = v;
  }
  cluster_sync(s.cs);
  if (warp == 0) {
    uint32_t c[1] = {0u};
    if (lane < kSlices) {  // lane i: slice kSlices - 1 - i
      const uint32_t* p = &sh.coarse[PASS][kSlices - 1 - lane];
      if (s.cs == 1) {
        c[0] = *p;
      } else {
#pragma unroll 8
        for (int r = 0; r < s.cs; ++r) c[0] += ld_peer(p, r);
      }
    }
    find_bin<1>(c, krem, [&](int i, uint32_t above, uint32_t) {
      sh.slice = (uint32_t)(kSlices - 1 - i);
      sh.above = above;
    });
  }
  if (s.cs > 1) {
    __syncthreads();
    // groups of threads, each adding some CTAs' counts of the slice's bins
    constexpr int kGroups = NT / kPer;
    const uint32_t* p = hist + sh.slice * kPer + tid % kPer;
    uint32_t t = 0u;
#pragma unroll 4
    for (int r = tid / kPer; r < s.cs; r += kGroups) t += ld_peer(p, r);
    sh.part[tid] = t;
    __syncthreads();
  }
  if (warp == 0) {
    __syncwarp();
    const int top = (int)(sh.slice + 1) * kPer - 1;
    uint32_t c[kLaneBins];
#pragma unroll
    for (int t = 0; t < kLaneBins; ++t) {
      const int bin = top - lane * kLaneBins - t;
      if (s.cs == 1) {
        c[t] = hist[bin];
      } else {
        c[t] = 0u;
#pragma unroll
        for (int g = 0; g < NT / kPer; ++g) c[t] += sh.part[g * kPer + bin % kPer];
      }
    }
    const uint32_t above = sh.above;
    find_bin<kLaneBins>(c, krem - above, [&](int i, uint32_t before, uint32_t count) {
      sh.digit = (uint32_t)(top - i);
      sh.before = above + before;
      sh.in_digit = count;
    });
  }
  __syncthreads();
  prefix |= sh.digit << pass_shift(PASS);
  krem -= sh.before;
  in_digit = sh.in_digit;
}

template <int NT>
__device__ __forceinline__ void clear(Shared<NT>& sh) {
  if (threadIdx.x == 0) {
    sh.slice = sh.above = sh.digit = sh.before = sh.in_digit = 0u;
    sh.jcut = INT_MAX;
  }
  for (int i = threadIdx.x; i < 4096; i += NT) sh.hist[i] = 0u;
}
// Pass 0's count of a key (the bound keeps any bit pattern inside the histogram).
__device__ __forceinline__ void count_key(uint32_t* hist, uint32_t x) {
  atomicAdd(&hist[min(x >> pass_shift(0), 2047u)], 1u);
}
template <int PASS, int NT, typename Key>
__device__ __forceinline__ void count_pass(Shared<NT>& sh, const Span& s, int end, uint32_t prefix, Key key) {
  constexpr uint32_t mask = PASS == 1 ? 0xFFF00000u : 0xFFFFFC00u;
#pragma unroll 4
  for (int i = s.wlo + (int)(threadIdx.x & 31); i < end; i += 32) {
    const uint32_t x = key(i);
    if (x != kNoKey && (x & mask) == prefix)
      atomicAdd(&sh.hist[pass_off(PASS) + ((x >> pass_shift(PASS)) & 1023u)], 1u);
  }
}

// The threshold (T, jcut) of the top-k of the keys below position hi, 0 < k < their number, digit pass 0
// already counted in sh.hist.  jcut: the last position taken among the keys equal to T.
template <int NT>
__device__ __forceinline__ void radix_select(Shared<NT>& sh, const Span& s, int hi, uint32_t k, uint32_t& T, int& jcut) {
  const int lane = threadIdx.x & 31, end = part_end(s, hi);
  auto key = [&](int i) { return s.base + i < hi ? s.keys[i] : kNoKey; };
  uint32_t prefix = 0u, krem = k, cnt = 0u;
  pick_digit<0>(sh, s, prefix, krem, cnt);
  count_pass<1>(sh, s, end, prefix, key);
  pick_digit<1>(sh, s, prefix, krem, cnt);
  count_pass<2>(sh, s, end, prefix, key);
  pick_digit<2>(sh, s, prefix, krem, cnt);
  T = prefix;
  jcut = INT_MAX;
  if (cnt != krem) {  // (the same in every CTA) more keys equal T than are needed: the lowest positions
    uint32_t eq = 0u, total;
    for (int i = s.wlo + lane; i < end; i += 32) eq += __popc(__ballot_sync(0xffffffffu, key(i) == T));
    uint32_t rank = scan_cluster(sh, s, 0, eq, total);
    for (int i = s.wlo + lane; i < end; i += 32) {
      const bool is = key(i) == T;
      const uint32_t bal = __ballot_sync(0xffffffffu, is);
      if (is && rank + __popc(bal & ((2u << lane) - 1u)) == krem)
        for (int r = 0; r < s.cs; ++r) {
          if (s.cs == 1) sh.jcut = s.base + i;
          else st_peer(reinterpret_cast<uint32_t*>(&sh.jcut), r, (uint32_t)(s.base + i));
        }
      rank += __popc(bal);
    }
    cluster_sync(s.cs);
    jcut = sh.jcut;
  }
}

// Kept flags and slots in position order (or their masks) and the kept positions of selection unit u: the selected
// keys below ncand and every position of the recent window [ncand, n).
template <int NT>
__device__ __forceinline__ void compact(const CompressArgs& a, Shared<NT>& sh, const Span& s, size_t u, int n, int ncand,
                                        int m, uint32_t T, int jcut) {
  const int lane = threadIdx.x & 31, end = part_end(s, n);
  auto kept_at = [&](int i) {
    const int j = s.base + i;
    if (j >= n) return false;
    if (j >= ncand) return true;
    const uint32_t x = s.keys[i];
    return x != kNoKey && (x > T || (x == T && j <= jcut));
  };
  uint32_t cnt = 0u, total;
  for (int i = s.wlo + lane; i < end; i += 32) cnt += __popc(__ballot_sync(0xffffffffu, kept_at(i)));
  uint32_t slot0 = scan_cluster(sh, s, 1, cnt, total);
  for (int i = s.wlo + lane; i < end; i += 32) {
    const bool kept = kept_at(i);
    const uint32_t bal = __ballot_sync(0xffffffffu, kept);
    const int j = s.base + i, slot = (int)(slot0 + __popc(bal & ((1u << lane) - 1u)));
    if (a.use_kmask && lane == 0) a.kmask[u * a.kmask_ld + (j >> 5)] = make_uint2(bal, slot0);
    slot0 += __popc(bal);
    if (j >= n) continue;
    if (!a.use_kmask) {
      a.kflag[u * a.n_cap + j] = kept ? 1 : 0;
      a.slot_of[u * a.n_cap + j] = kept ? slot : -1;
    }
    // with the full cosine routing: the evicted positions in order (slot = kept ones before j)
    if (!kept && a.routing == SELKV_ROUTE_COSINE) a.ev_pos[u * a.n_cap + (j - slot)] = j;
    if (kept && slot < a.m_cap) {
      a.kept_pos[u * a.m_cap + slot] = j;
      if (a.dbg_kept_idx != nullptr) a.dbg_kept_idx[u * a.m_cap + slot] = j;
    }
  }
  if (s.rank == 0 && threadIdx.x == 0 && (int)total != m) raise_flag(a.flags, SELKV_DEVERR_COUNT);
}

// Pooling of Eq. 1's score and each KV head's top-m_s.  Grid (cluster size, B * Hkv).  POOL is
// the pooling kernel (0: any, from the arguments).
template <int POOL, int NT>
__global__ __launch_bounds__(NT) void topk_kernel(CompressArgs a, SelectWs w, int near_keys) {
  chain_begin();
  cluster_started_arrive(gridDim.x);
  __shared__ Shared<NT> sh;
  extern __shared__ uint32_t dyn_keys[];
  const int u = blockIdx.y, b = u / a.Hkv, lane = threadIdx.x & 31;
  const int n = a.seq_n[b], ncand = n - a.recent, k = a.seq_m[b] - a.recent;
  float* sc = a.score + (size_t)u * a.n_cap;
  const Span s = make_span<NT>(n, gridDim.x, near_keys ? dyn_keys : nullptr, reinterpret_cast<uint32_t*>(sc));
  const bool narrow = k > 0 && k < ncand;
  clear(sh);
  __syncthreads();
  const int pool = POOL ? POOL : a.pool_kernel, half = pool / 2;
  const float* at = a.attn + (size_t)u * a.n_cap;
  const float* vn = a.vnorm + (size_t)u * a.n_cap;
  const int end = part_end(s, n);
  // Four steps at a time: their own two values are loaded together, and by the time a step
  // comes its neighbours' lines are in L1 too.
  constexpr int kAhead = 4;
  for (int g0 = s.wlo; g0 < end; g0 += 32 * kAhead) {
    float own_a[kAhead], own_v[kAhead];
#pragma unroll
    for (int p = 0; p < kAhead; ++p) {
      const int j = s.base + g0 + p * 32 + lane;
      own_a[p] = j < ncand ? at[j] : 0.f;
      own_v[p] = j < ncand ? vn[j] : 0.f;
    }
    float pooled[kAhead];  // (all of them before the first store, which a later load might depend on)
#pragma unroll
    for (int p = 0; p < kAhead; ++p) {
      const int i0 = g0 + p * 32, j = s.base + i0 + lane;
      float v = 0.f;
      if (POOL && s.base + i0 >= half && s.base + i0 + 31 + half < ncand) {  // every tap of the warp's positions
        const float *pa = at + j, *pv = vn + j;
#pragma unroll
        for (int t = -(POOL / 2); t <= POOL / 2; ++t)
          v = t == 0 ? fmaf(own_a[p], own_v[p], v) : fmaf(pa[t], pv[t], v);
      } else if (j < ncand) {
        for (int jj = max(0, j - half); jj <= min(ncand - 1, j + half); ++jj)
          v = fmaf(at[jj], vn[jj], v);
      }
      pooled[p] = v / (float)pool;
    }
#pragma unroll
    for (int p = 0; p < kAhead; ++p) {
      const int i0 = g0 + p * 32, i = i0 + lane, j = s.base + i;
      if (i0 >= end) break;  // the rest belongs to the next warp
      const float v = pooled[p];
      if (narrow && j < ncand) count_key(sh.hist, __float_as_uint(v));
      if (j < n) sc[j] = v;
      if (near_keys) s.keys[i] = __float_as_uint(v);
    }
  }
  cluster_started_wait(s.cs);
  uint32_t T = 0u;  // select every candidate ...
  int jcut = INT_MAX;
  if (k <= 0) {
    T = 0xffffffffu;  // ... or none
    jcut = -1;
  } else if (narrow) {
    radix_select(sh, s, ncand, (uint32_t)k, T, jcut);
  }
  if (!a.per_head) {
    if (s.rank == 0 && threadIdx.x == 0) w.topk[u] = RadixCut{T, jcut};
  } else {
    if (a.dbg_topk != nullptr)
      for (int i = s.wlo + lane; i < end; i += 32) {
        const int j = s.base + i;
        if (j < n) a.dbg_topk[(size_t)u * a.n_cap + j] = j < ncand && (s.keys[i] > T || (s.keys[i] == T && j <= jcut));
      }
    compact(a, sh, s, u, n, ncand, a.seq_m[b], T, jcut);
  }
  cluster_sync(s.cs);  // no CTA leaves while another may still read its shared memory
}

// Union over KV heads, trimmed to m_s by the score summed over KV heads, then the compaction.
// Grid (cluster size, B).
template <int NT>
__global__ __launch_bounds__(NT) void trim_kernel(CompressArgs a, SelectWs w, int near_keys) {
  chain_begin();
  cluster_started_arrive(gridDim.x);
  __shared__ Shared<NT> sh;
  __shared__ RadixCut cut[32];
  extern __shared__ uint32_t dyn_keys[];
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int n = a.seq_n[b], ncand = n - a.recent, k = a.seq_m[b] - a.recent;
  const Span s = make_span<NT>(n, gridDim.x, near_keys ? dyn_keys : nullptr, w.tkey + (size_t)b * a.n_cap);
  clear(sh);
  if ((int)threadIdx.x < a.Hkv) cut[threadIdx.x] = w.topk[(size_t)b * a.Hkv + threadIdx.x];
  __syncthreads();
  const int end = part_end(s, n);
  const float* sc0 = a.score + (size_t)b * a.Hkv * a.n_cap;
  uint32_t cnt = 0u, members;
  // Score of head h at position j, and whether j is in the head's top-m_s.  Ties at a head's
  // threshold are rare: without any, one comparison decides.
  const bool ties = __syncthreads_or((int)threadIdx.x < a.Hkv && cut[threadIdx.x].jcut != INT_MAX);
  constexpr int kHeads = 8, kAhead = 2;  // scores loaded together: of kHeads heads, kAhead steps
  const size_t stride = (size_t)a.n_cap;
  for (int g0 = s.wlo; g0 < end; g0 += 32 * kAhead) {
    bool in[kAhead];
    float sum[kAhead];
#pragma unroll
    for (int p = 0; p < kAhead; ++p) {
      in[p] = false;
      sum[p] = 0.f;
    }
    const int j0 = s.base + g0 + lane;
    const float* row = sc0 + j0;
    for (int kv0 = 0; kv0 < a.Hkv; kv0 += kHeads, row += kHeads * stride) {
      const int nh = min(kHeads, a.Hkv - kv0);
      float v[kAhead][kHeads];
#pragma unroll
      for (int p = 0; p < kAhead; ++p)
#pragma unroll
        for (int h = 0; h < kHeads; ++h)
          v[p][h] = h < nh && j0 + p * 32 < n ? row[h * stride + p * 32] : 0.f;
#pragma unroll
      for (int h = 0; h < kHeads; ++h) {
        if (h >= nh) break;
        const RadixCut c = cut[kv0 + h];
#pragma unroll
        for (int p = 0; p < kAhead; ++p) {
          const uint32_t x = __float_as_uint(v[p][h]);
          in[p] |= ties ? x > c.T || (x == c.T && j0 + p * 32 <= c.jcut) : x >= c.T;
          sum[p] += v[p][h];
        }
      }
    }
#pragma unroll
    for (int p = 0; p < kAhead; ++p) {
      const int i0 = g0 + p * 32, i = i0 + lane, j = s.base + i;
      if (i0 >= end) break;  // the rest belongs to the next warp
      const bool member = in[p] && j < ncand;
      if (near_keys || j < ncand) s.keys[i] = member ? __float_as_uint(sum[p]) : kNoKey;
      if (member) count_key(sh.hist, __float_as_uint(sum[p]));
      cnt += __popc(__ballot_sync(0xffffffffu, member));
    }
  }
  if (a.dbg_topk != nullptr)
    for (int i = s.wlo + lane; i < end; i += 32) {
      const int j = s.base + i;
      for (int kv = 0; kv < a.Hkv && j < n; ++kv) {
        const uint32_t x = __float_as_uint(sc0[(size_t)kv * a.n_cap + j]);
        a.dbg_topk[((size_t)b * a.Hkv + kv) * a.n_cap + j] =
            j < ncand && (x > cut[kv].T || (x == cut[kv].T && j <= cut[kv].jcut));
      }
    }
  cluster_started_wait(s.cs);
  scan_cluster(sh, s, 0, cnt, members);
  uint32_t T = 0u;
  int jcut = INT_MAX;
  if ((int)members > k) radix_select(sh, s, ncand, (uint32_t)k, T, jcut);  // (k > 0: no member otherwise)
  compact(a, sh, s, b, n, ncand, a.seq_m[b], T, jcut);
  cluster_sync(s.cs);  // no CTA leaves while another may still read its shared memory
}

// CTAs per selection: a power of two, doubled while the selections leave SMs without a CTA and a
// CTA would hold more than 1024 positions.  Up to 16 for a few selections; more of them take 8 at
// most, since CTAs of 1024 threads leave room for 7 clusters of 16 only (8 heads x 100k: topk 18.9 us
// with 8, 20.6 with 16 CTAs of 512 threads).
int cluster_size(int units, int n_cap) {
  const int most = units > 4 ? 8 : kMaxCluster;
  int cs = 1;
  while (cs < most && units * cs < kPlanSMs && n_cap > 1024 * cs) cs *= 2;
  return cs;
}
// 1024 threads a CTA where the CTAs leave SMs empty and each has two warps' worth of steps or
// more: what takes the time there is a warp's own steps (one sequence of 100k: trim 27.3 -> 23.0
// us).  Where CTAs share an SM, 512 (64 x 8k, the same).
bool wide_ctas(int units, int n_cap) {
  const int cs = cluster_size(units, n_cap);
  return units * cs <= 100 && n_cap > 512 * cs;
}

// The largest cluster of the kernel's CTAs, with the most shared memory they take, that the device can
// place, looked up once per kernel and device.  Sixteen CTAs need as many free SMs in one GPC, which a
// partition of the GPU may not have; the selection is the same for every cluster size.
template <auto Kern, int NT>
int largest_cluster() {
  static std::atomic<int> found[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  int cs = found[dev].load(std::memory_order_acquire);
  if (cs > 0) return cs;
  cs = fit_cluster(kMaxCluster, [](int size) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = kMaxSpan * 4;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, Kern, &cfg) == cudaSuccess) return clusters > 0;
    cudaGetLastError();  // (a refusal is an answer, not an error of the call)
    return false;
  });
  found[dev].store(cs, std::memory_order_release);
  return cs;
}

template <auto Kern, int NT>
cudaError_t launch_clusters(const CompressArgs& a, const SelectWs& w, int units, int want, cudaStream_t s) {
  cudaError_t e = set_smem_once<Kern>(kMaxSpan * 4);
  if (e == cudaSuccess) e = allow_any_cluster_once<Kern>();
  if (e != cudaSuccess) return e;
  const int cs = std::min(want, largest_cluster<Kern, NT>());
  const int span = ((a.n_cap + cs - 1) / cs + NT - 1) / NT * NT;
  const int near_keys = span <= kMaxSpan ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, units);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = near_keys ? (size_t)span * 4 : 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // (as launch_chained)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.chain ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, Kern, a, w, near_keys);
}

}  // namespace

size_t select_ws_bytes(int B, int Hkv, int n_cap) {
  const size_t units = (size_t)B * Hkv;
  return units * sizeof(RadixCut) + (size_t)B * n_cap * 4 + 2 * 256;  // two regions, each rounded up to 256 bytes
}

SelectWs carve_select_ws(void* base, int B, int Hkv, int n_cap) {
  const size_t units = (size_t)B * Hkv;
  SelectWs w{};
  w.topk = static_cast<RadixCut*>(base);
  w.tkey = reinterpret_cast<uint32_t*>(static_cast<char*>(base) + ((units * sizeof(RadixCut) + 255) & ~size_t(255)));
  return w;
}

// Pooling and the whole selection: 2 kernels (1 in the per-head mode), no host sync.
cudaError_t launch_select_grid(const CompressArgs& a, const SelectWs& w, cudaStream_t s) {
  auto topk = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    const int units = a.B * a.Hkv, cs = cluster_size(units, a.n_cap);
    return a.pool_kernel == 5 ? launch_clusters<topk_kernel<5, NT>, NT>(a, w, units, cs, s)
                              : launch_clusters<topk_kernel<0, NT>, NT>(a, w, units, cs, s);
  };
  auto trim = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    return launch_clusters<trim_kernel<NT>, NT>(a, w, a.B, cluster_size(a.B, a.n_cap), s);
  };
  using Few = std::integral_constant<int, 512>;
  using Many = std::integral_constant<int, 1024>;
  cudaError_t e = wide_ctas(a.B * a.Hkv, a.n_cap) ? topk(Many{}) : topk(Few{});
  if (e == cudaSuccess && !a.per_head) e = wide_ctas(a.B, a.n_cap) ? trim(Many{}) : trim(Few{});
  return e;
}

}  // namespace selkv
