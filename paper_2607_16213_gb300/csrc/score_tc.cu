// Observation-window scoring on the 5th-generation tensor cores (bf16 caches).
//
// Per (sequence b, KV head kv) the G query heads' W window rows are stacked into R = G W rows
// (row r = g W + i is query head kv G + g at position p = n_b - W + i, which sees keys j <= p:
// the causal re-pass of Sec. 3.1).  With s'_rj = log2(e) q_r . k_j / sqrt(d):
//   pass 1: per row, over a slice of the keys: (max_j s'_rj, sum_j 2^(s'_rj - max)),
//   pass 2: M_r, Z_r over the slices, then
//           a_j = sum_r 2^(s'_rj - M_r) / (G Z_r) = sum_r 2^(s'_rj - M_r - log2(G Z_r))
//           (Eq. 5's a, mean over the group).
// Both passes are one kernel: a TMA producer warp streams K tiles (and the group's Q once)
// into shared memory with 128-byte swizzling; one thread issues tcgen05.mma (bf16 in, fp32
// accumulate, N = 256 so each instruction carries a full-width product) into one of two
// tensor-memory accumulators; sixteen epilogue warps (four per scheduler) read the
// accumulator with tcgen05.ld and reduce it while the next tile is multiplied.  Pass 1 puts
// 128 query rows in the accumulator lanes (M = 128) and 256 keys in its columns; a CTA owns 128
// rows, or two such halves in turn on the same keys; an epilogue thread owns a row (of each half) and
// a quarter of each tile's keys, and the four quarter states of a row are folded at the end.  Pass 2 puts 128 keys in
// the lanes and the R rows in the columns; an epilogue thread owns a key and a quarter of the
// rows, and the four quarters' column sums of a key are added in shared memory in a fixed
// order before a_j is written.
//
// Every wait is bounded; on timeout the CTA raises SELKV_DEVERR_TIMEOUT, keeps the barrier
// protocol of its epilogue warps, lets issued copies and MMAs finish (bounded) and frees its
// tensor memory before leaving.
#include <cudaTypedefs.h>

#include <type_traits>

#include "ptx.cuh"
#include "selkv_internal.cuh"

namespace selkv {
namespace {

constexpr uint32_t kTmemCols = 512;  // two accumulators of up to 256 fp32 columns
#ifndef SELKV_P1_KEYS
#define SELKV_P1_KEYS 256  // pass 1: keys per tile (the MMA's N), a multiple of 32
#endif
#ifndef SELKV_P1_CPW
#define SELKV_P1_CPW 2     // pass 1: 32-column accumulator chunks per epilogue warp and tile
#endif
constexpr int kP2Keys = 128;  // pass 2: keys per tile
// Epilogue warps: pass 1 splits a tile's keys over the warps of each TMEM lane quarter (32
// columns x SELKV_P1_CPW per warp), pass 2 splits the rows over four warps per lane quarter.
// A TMA producer warp and an MMA warp follow them.
constexpr int kP1Parts = SELKV_P1_KEYS / (32 * SELKV_P1_CPW);
static_assert(kP1Parts * 32 * SELKV_P1_CPW == SELKV_P1_KEYS && kP1Parts >= 1, "pass-1 tile split");
// Both passes also carry the value norms of Eq. 1 (selkv_compress only) in a few more warps, half
// of the rows each.  A kernel of its own for them, whether before the passes or beside them on
// another stream, took all SMs first and cost its whole time (58 us for one layer of 8 x 100k
// rows); the passes have room for its bytes: 50 + 53 us become 53 + 55.  All rows in pass 1 make it
// wait for HBM (68 + 58 us with one row half per CTA), all in pass 2 wait for the three warps of
// two copies in flight that its shared memory holds (50 + 78); shares of 3/8 and 5/8 in pass 1 are
// within 2% of halves.  Two warps with as many bytes in flight are too slow (59 + 60 us).
__host__ __device__ constexpr int norm_warps(int pass, int halves) { return pass == 1 && halves == 1 ? 4 : 3; }
__host__ __device__ constexpr int norm_stages(int pass, int halves) { return pass == 1 && halves == 1 ? 3 : 2; }
static_assert(4 * kP1Parts + 2 + norm_warps(1, 1) <= 32 && SELKV_P1_KEYS <= 256, "pass-1 warps per CTA");
__host__ __device__ constexpr int epi_warps(int pass) { return pass == 1 ? 4 * kP1Parts : 16; }
__host__ __device__ constexpr int cta_threads(int pass, int halves, bool norms) {
  return (epi_warps(pass) + 2 + (norms ? norm_warps(pass, halves) : 0)) * 32;
}

// Value norms of rows [row_lo, row_hi) by warp `w` of norm_warps.  The rows of a (sequence,
// KV head) are contiguous, so lane 0 streams them as 4 KB bulk copies into the warp's own ring
// (bytes in flight cost no registers; with 4 KB in registers per warp the round trips of eight
// warps made pass 1 277 us for 64 x 8k where this took 235).  D / 8 lanes take a row, 16 bytes a
// lane: a lane squares its 8 elements in order and the lanes of a row meet in a butterfly; the
// sums of a chunk's 8 row groups share it (each level keeps half of the values), pairing the
// lanes as a butterfly per value does.  The copies are marked for early eviction from L2.
constexpr int kNormChunk = 4096;  // bytes per copy
__host__ __device__ constexpr int norm_ring(int pass, int halves) {
  return norm_warps(pass, halves) * norm_stages(pass, halves) * kNormChunk;
}
// `used` counts the copies this warp has taken from its ring; false after a timed-out wait.
template <int D, int PASS, int HALVES>
__device__ __forceinline__ bool norm_rows(const __nv_bfloat16* V, float* norm, int row_lo, int row_hi, int w,
                                          unsigned char* ring, uint64_t* bars, uint32_t* flags, int& used) {
  constexpr int LPR = D / 8, RPL = 32 / LPR, kGroups = kNormChunk / 512;  // lanes per row, rows per group of lanes
  constexpr int kNormStages = norm_stages(PASS, HALVES), nw = norm_warps(PASS, HALVES);
  constexpr int kRows = RPL * kGroups;                     // rows per chunk
  static_assert(kRows * D * 2 == kNormChunk, "a chunk is whole rows");
  const int lane = threadIdx.x & 31, sub = lane / LPR;
  ring += w * kNormStages * kNormChunk;
  bars += w * kNormStages;
  const int first = row_lo + w * kRows, stride = nw * kRows;
  const int chunks = first < row_hi ? (row_hi - first + stride - 1) / stride : 0;
  const uint64_t pol = l2_evict_first_policy();
  auto load = [&](int c) {
    const int r0 = first + c * stride, st = (used + c) % kNormStages;
    const uint32_t bytes = (uint32_t)min(kRows, row_hi - r0) * D * 2;
    mbar_arrive_expect_tx(&bars[st], bytes);
    bulk_load_hint(ring + st * kNormChunk, V + (size_t)r0 * D, bytes, &bars[st], pol);
  };
  if (lane == 0)
    for (int c = 0; c < min(chunks, kNormStages); ++c) load(c);
  for (int c = 0; c < chunks; ++c) {
    const int st = (used + c) % kNormStages, r0 = first + c * stride;
    if (!__all_sync(0xffffffffu, mbar_wait(&bars[st], ((used + c) / kNormStages) & 1))) {
      if (lane == 0) {
        raise_flag(flags, SELKV_DEVERR_TIMEOUT);
        for (int k = c; k < min(chunks, c + kNormStages); ++k)  // (bounded) let the copies in flight land
          mbar_wait(&bars[(used + k) % kNormStages], ((used + k) / kNormStages) & 1);
      }
      return false;
    }
    const uint4* src = reinterpret_cast<const uint4*>(ring + st * kNormChunk) + lane;
    float q[kGroups];
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
      const uint4 u = src[k * 32];
      const uint32_t x[4] = {u.x, u.y, u.z, u.w};
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = bf16_lo(x[e]), hi = bf16_hi(x[e]);
        s = fmaf(lo, lo, s);
        s = fmaf(hi, hi, s);
      }
      q[k] = s;
    }
    __syncwarp();
    if (lane == 0 && c + kNormStages < chunks) load(c + kNormStages);
    int k0 = 0;  // first group whose sum this lane still holds; `keep` of them follow
#pragma unroll
    for (int o = LPR / 2, keep = kGroups; o > 0; o >>= 1) {
      const bool up = lane & o;
      if (keep > 1) {
        keep >>= 1;
#pragma unroll
        for (int i = 0; i < keep; ++i) {
          const float mine = up ? q[keep + i] : q[i], other = up ? q[i] : q[keep + i];
          q[i] = mine + __shfl_xor_sync(0xffffffffu, other, o);
        }
        k0 += up ? keep : 0;
      } else {
        q[0] += __shfl_xor_sync(0xffffffffu, q[0], o);
      }
    }
    // LPR lanes hold kGroups sums: the lowest of the lanes that share one writes it
    const int row = r0 + k0 * RPL + sub;
    if ((lane % (LPR / kGroups)) == 0 && row < row_hi) norm[row] = sqrtf(q[0]);
  }
  used += chunks;
  return true;
}

#ifndef SELKV_P2_PIPE
#define SELKV_P2_PIPE 1   // pass 2: pipelined 16-column TMEM loads on full, unmasked tiles
#endif

// Pass 2, one thread's key over 64 rows of a tile (no causal mask): the sum over the rows of
// 2^(v sc - M_r - log2(G Z_r)).  The accumulator is read 16 columns at a time, each load
// issued before the arithmetic on the previous one so its latency overlaps that work; row
// pairs are packed (f32x2) and summed in four interleaved partial sums.
__device__ __forceinline__ void colsum_accum16(const float (&v)[16], uint32_t rn, uint64_t sc2,
                                               uint64_t& a01, uint64_t& a23) {
#pragma unroll
  for (int i = 0; i < 16; i += 4) {
    const float4 nm = lds_f4(rn + i * 4);  // -(M + log2(G Z)) of rows i .. i+3
    float x0, x1, x2, x3;
    unpack_f2(ffma2(pack_f2(v[i], v[i + 1]), sc2, pack_f2(nm.x, nm.y)), x0, x1);
    unpack_f2(ffma2(pack_f2(v[i + 2], v[i + 3]), sc2, pack_f2(nm.z, nm.w)), x2, x3);
    a01 = fadd2(a01, pack_f2(ex2_approx(x0), ex2_approx(x1)));
    a23 = fadd2(a23, pack_f2(ex2_approx(x2), ex2_approx(x3)));
  }
}
__device__ __forceinline__ float colsum64(uint32_t taddr, uint32_t rn, float sc) {
  const uint64_t sc2 = pack_f2(sc, sc);
  uint64_t a01 = pack_f2(0.f, 0.f), a23 = a01;
  float va[16], vb[16];
  tmem_ld16_issue(taddr, va);
  tmem_wait_ld16(va);
#pragma unroll
  for (int c = 0; c < 4; c += 2) {
    tmem_ld16_issue(taddr + (c + 1) * 16, vb);
    colsum_accum16(va, rn + c * 64, sc2, a01, a23);
    tmem_wait_ld16(vb);
    if (c + 2 < 4) tmem_ld16_issue(taddr + (c + 2) * 16, va);
    colsum_accum16(vb, rn + (c + 1) * 64, sc2, a01, a23);
    if (c + 2 < 4) tmem_wait_ld16(va);
  }
  float s0, s1, s2, s3;
  unpack_f2(a01, s0, s1);
  unpack_f2(a23, s2, s3);
  return (s0 + s1) + (s2 + s3);
}

// HALVES (pass 2): 1 when the R rows fit one accumulator of 256 columns, 2 when they take two
// (R up to 512): each key tile is then multiplied by the two 256-row halves of Q in turn, the
// halves alternating between the two accumulators, and the K ring is shortened to make room
// for the 512 staged rows.
template <int D, int PASS, int HALVES = 1>
struct SCfg {
  static constexpr int kKeys = PASS == 1 ? SELKV_P1_KEYS : kP2Keys;    // keys per tile
  static constexpr int kStages = PASS == 1 ? 2 : (HALVES == 2 ? 2 : 4);  // K tiles in flight
  static constexpr int kRows = (PASS == 1 ? 128 : 256) * HALVES;        // Q rows staged per CTA
  static constexpr int kBoxes = D / 64;                  // 128-byte-wide boxes per row
  static constexpr int kKTile = kKeys * D * 2;           // one K tile
  static constexpr int kQBytes = kRows * D * 2;
  static constexpr int kRing = kStages * kKTile;
  // barriers | -(M + log2(G Z)) and window place of up to 512 rows | pass 1: [parts][128] float2, pass 2: [2][4][128] float
  static constexpr int kHead = 384;  // barriers and flags
  static constexpr int kMisc = kHead + (PASS == 1 ? 0 : 512 * 8) + (kP1Parts * 128 * 8 > 4096 ? kP1Parts * 128 * 8 : 4096);
  static constexpr int kSmem = 1024 + kQBytes + kRing + kMisc + norm_ring(PASS, HALVES);
  static_assert(kSmem <= 232448, "227 KB of shared memory");
};

// One CTA's share of a pass: `cnt` consecutive key tiles of the list of all (unit, tile) pairs, in
// unit order (unit = sequence b, KV head kv), as pieces of one unit each.  Every role of the CTA
// walks the same pieces.
struct Walk {
  int u, t, left;              // the piece's unit and first tile, tiles left from there
  int b, kv, n, ntiles, nt;    // its sequence, head and length; the unit's tiles; the piece's tiles
  __device__ __forceinline__ void open(const CompressArgs& a, int keys, int len = 0) {
    if (left <= 0) return;
    b = u / a.Hkv;
    kv = u - b * a.Hkv;
    n = len > 0 ? len : a.seq_n[b];
    ntiles = (n + keys - 1) / keys;
    nt = min(left, ntiles - t);
  }
  __device__ __forceinline__ void next(const CompressArgs& a, int keys) {
    left -= nt;
    ++u;
    t = 0;
    open(a, keys);
  }
};

// The partials that pass 1 left of unit u (T1 of its tiles, the first one `before` tiles into the list
// of all): one from each CTA group that held tiles of it, at first .. first + count - 1.
struct Partials {
  int first, count;
};
__host__ __device__ __forceinline__ Partials partials_of(int split, int per, int u, int before, int T1) {
  int c0, c1;
  if (split > 0) {
    const int p = (T1 + split - 1) / split;
    c0 = u * split;
    c1 = c0 + (T1 - 1) / p;
  } else {
    c0 = before / per;
    c1 = (before + T1 - 1) / per;
  }
  return {c0 + u, c1 - c0 + 1};
}
__device__ __forceinline__ Partials partials_of(const CompressArgs& a, const ScoreWalk& s, const Walk& w) {
  const int T1 = (w.n + SELKV_P1_KEYS - 1) / SELKV_P1_KEYS;
  return partials_of(s.p1_split, s.p1_per, w.u, s.p1_split > 0 ? 0 : a.seq_t1[w.b] * a.Hkv + w.kv * T1, T1);
}

// Fold of the partials of row r: -(M + log2(G Z)), the row's whole normaliser as one exponent offset
// (2^(s' - M) / (G Z) = 2^(s' - (M + log2(G Z)))).
__device__ __forceinline__ float fold_row_tc(const CompressArgs& a, const Partials& ps, int r) {
  const float2* part = a.rowpart + (size_t)ps.first * a.R + r;
  const int nch = ps.count;
  float M = -INFINITY, Z = 0.f;
  constexpr int kAhead = 8;  // partials loaded together
  for (int c = 0; c < nch; c += kAhead) {
    float2 p[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
      p[i] = c + i < nch ? part[(size_t)(c + i) * a.R] : make_float2(-INFINITY, 0.f);
    float m = M;
#pragma unroll
    for (int i = 0; i < kAhead; ++i) m = fmaxf(m, p[i].x);
    if (m == -INFINITY) continue;
    Z *= exp2f(M - m);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) Z += p[i].y * exp2f(p[i].x - m);
    M = m;
  }
  const float y = 1.f / ((float)a.G * Z);
  return y > 0.f ? -(M - log2f(y)) : -INFINITY;
}

// Pass 1: the sum of 2^(v sc - ref) over a row's 32 keys; pairs packed, four interleaved partial sums.
__device__ __forceinline__ float rowsum32(const float (&v)[32], float sc, float ref) {
  const uint64_t sc2 = pack_f2(sc, sc), nm2 = pack_f2(-ref, -ref);
  uint64_t s01 = pack_f2(0.f, 0.f), s23 = s01;
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    float x0, x1, x2, x3;
    unpack_f2(ffma2(pack_f2(v[i], v[i + 1]), sc2, nm2), x0, x1);
    unpack_f2(ffma2(pack_f2(v[i + 2], v[i + 3]), sc2, nm2), x2, x3);
    s01 = fadd2(s01, pack_f2(ex2_approx(x0), ex2_approx(x1)));
    s23 = fadd2(s23, pack_f2(ex2_approx(x2), ex2_approx(x3)));
  }
  float s0, s1, s2, s3;
  unpack_f2(s01, s0, s1);
  unpack_f2(s23, s2, s3);
  return (s0 + s1) + (s2 + s3);
}

// TABLE (pass 2 in a call of its own): the shares are those that the call with pass 1 left in the
// workspace, which go with its lengths there; otherwise they come with the launch.
template <int D, int PASS, int HALVES, bool TABLE = false>
__global__ __launch_bounds__(cta_threads(PASS, HALVES, true), 1) void score_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                                        const __grid_constant__ CUtensorMap tmK,
                                                                        CompressArgs a,
                                                                        const __grid_constant__ ScoreWalk shares) {
  using C = SCfg<D, PASS, HALVES>;
  constexpr int kEpiWarps = epi_warps(PASS);
  constexpr int kProducerWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1;
  constexpr int kKeys = C::kKeys, kStages = C::kStages;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* Qs = smem;                  // [kBoxes][Rq rows][128 B]
  unsigned char* Ks = smem + C::kQBytes;     // [kStages][kBoxes][kKeys rows][128 B]
  unsigned char* misc = Ks + C::kRing;
  uint64_t* full = reinterpret_cast<uint64_t*>(misc);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* qbar = tempty + 2;    // the piece's Q is in
  uint64_t* qfree = qbar + 1;     // the piece's MMAs have read it
  uint64_t* done = qfree + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // pass 2: per lane quarter and column-sum buffer, "the other three parts' sums are in" and
  // "part 0 has read them"
  uint64_t* cs_full = reinterpret_cast<uint64_t*>(misc + 128);  // [4][2]
  uint64_t* cs_empty = cs_full + 8;                              // [4][2]
  // the norm warps' copies, and their ring
  static_assert((2 * kStages + 7) * 8 + 8 <= 128, "barriers and flags before the column sums'");
  constexpr int kNormBars = norm_warps(PASS, HALVES) * norm_stages(PASS, HALVES);
  static_assert(kNormBars <= 16, "norm barriers fit");
  uint64_t* nbar = reinterpret_cast<uint64_t*>(misc + 256);
  unsigned char* nring = misc + C::kMisc;
  float* rneg = reinterpret_cast<float*>(misc + C::kHead);               // pass 2: -(M + log2(G Z)) per row
  int* rwin = reinterpret_cast<int*>(misc + C::kHead + 512 * 4);         // pass 2: r mod W per row, its place in the window
  float* colpart = reinterpret_cast<float*>(misc + C::kHead + (PASS == 1 ? 0 : 512 * 8));  // pass 1: [parts][128] float2; pass 2: [2][4][128]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int R = a.R;
  const int Rp = (R + 15) & ~15;              // N of the pass-2 MMAs over all halves
  constexpr int kP1Rows = 128 * HALVES;
  const int MT = (R + kP1Rows - 1) / kP1Rows;  // pass 1: row parts of the R rows, a CTA each
  const int h = PASS == 1 ? (int)blockIdx.x % MT : 0;           // pass 1: this CTA's rows
  const int group = PASS == 1 ? (int)blockIdx.x / MT : (int)blockIdx.x;  // CTAs with the same tiles
  const int nph = PASS == 1 ? min(HALVES, (R - h * kP1Rows + 127) / 128) : HALVES;  // row halves in use
  const int Rq = PASS == 1 ? kP1Rows : (HALVES == 2 ? 512 : (R > 128 ? 256 : 128));  // Q rows staged (whole boxes)
  const ScoreWalk& walk = TABLE ? *a.p2_walk : shares;
  Walk w0{walk.u0[group], walk.t0[group], walk.cnt[group], 0, 0, 0, 0, 0};
  w0.open(a, kKeys, walk.n[group]);

  // Loads of the producer's lane 0: a tile of keys, and the rows of the piece's Q.
  auto load_tile = [&](const Walk& w, int t, int st) {
    const int krow0 = (int)((size_t)w.u * a.n_cap) + w.t * kKeys;
    mbar_arrive_expect_tx(&full[st], C::kKTile);
    for (int bx = 0; bx < C::kBoxes; ++bx)
      tma_load_2d(Ks + st * C::kKTile + bx * kKeys * 128, &tmK, bx * 64, krow0 + t * kKeys, &full[st]);
  };
  auto load_q = [&](const Walk& w) {
    const int qrow0 = (w.b * a.Hq + w.kv * a.G) * a.W + h * kP1Rows;
    mbar_arrive_expect_tx(qbar, C::kBoxes * Rq * 128);
    for (int bx = 0; bx < C::kBoxes; ++bx)
      for (int r0 = 0; r0 < Rq; r0 += 128) tma_load_2d(Qs + (bx * Rq + r0) * 128, &tmQ, bx * 64, qrow0 + r0, qbar);
  };
  const int early = w0.left > 0 ? min(kStages, w0.nt) : 0;  // tiles loaded before the CTA is set up
  if (threadIdx.x == kProducerWarp * 32) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], kEpiWarps);
    }
    mbar_init(qbar, 1);
    mbar_init(qfree, 1);
    mbar_init(done, 1);
    for (int i = 0; i < kNormBars; ++i) mbar_init(&nbar[i], 1);
    if (PASS == 2) {
      for (int i = 0; i < 8; ++i) {
        mbar_init(&cs_full[i], 3);
        mbar_init(&cs_empty[i], 1);
      }
    }
    *abort_flag = 0;
    fence_mbar_init();
    // Q and the first tiles at once: K and Q are inputs of the call, complete before its first kernel
    // starts, whatever the kernel before this one still does.
    prefetch_tensormap(&tmQ);
    prefetch_tensormap(&tmK);
    if (early > 0) {
      load_tile(w0, 0, 0);
      load_q(w0);
      for (int t = 1; t < early; ++t) load_tile(w0, t, t);
    }
  }
  __syncwarp();
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, kTmemCols);
  chain_begin();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == kProducerWarp) {
    if (lane == 0) {
      int tt = 0;      // tiles issued, over all pieces
      int pieces = 0;  // pieces whose Q is issued
      bool ok = true;
      for (Walk w = w0; ok && w.left > 0; w.next(a, kKeys)) {
        for (int t = 0; t <= w.nt; ++t) {
          // Q after the piece's first tile, which can be loaded while the last piece's MMAs still read theirs
          if (t == 1) {
            if (pieces > 0) {
              if (!mbar_wait(qfree, (pieces - 1) & 1) || *abort_flag) {
                ok = false;
                break;
              }
              load_q(w);
            }
            ++pieces;  // (the first piece's was loaded above)
          }
          if (t == w.nt) break;
          if (tt >= early) {
            const int st = tt % kStages;
            if (!mbar_wait(&empty[st], ((tt / kStages) & 1) ^ 1) || *abort_flag) {
              ok = false;
              break;
            }
            load_tile(w, t, st);
          }
          ++tt;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
      }
      for (int t = max(0, tt - kStages); t < tt; ++t) mbar_wait(&full[t % kStages], (t / kStages) & 1);
      if (pieces > 0) mbar_wait(qbar, (pieces - 1) & 1);
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0 && w0.left > 0) {
      bool ok = true;
      const uint32_t qbase = smem_u32(Qs);
      int u = 0;   // accumulator use: one per (key tile, row half)
      int tt = 0;  // tiles, over all pieces
      int pieces = 0;
      for (Walk w = w0; ok && w.left > 0; w.next(a, kKeys), ++pieces) {
        ok = mbar_wait(qbar, pieces & 1) && !*abort_flag;
        for (int t = 0; ok && t < w.nt; ++t, ++tt) {
          const int st = tt % kStages;
          if (!mbar_wait(&full[st], (tt / kStages) & 1) || *abort_flag) {
            ok = false;
            break;
          }
          const uint32_t kbase = smem_u32(Ks + st * C::kKTile);
          for (int ph = 0; ph < nph; ++ph, ++u) {
            const int buf = u & 1;
            if (!mbar_wait(&tempty[buf], ((u >> 1) & 1) ^ 1) || *abort_flag) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t idesc = PASS == 1 ? umma_idesc_bf16(128, kKeys) : umma_idesc_bf16(128, min(256, Rp - ph * 256));
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t koff = (ks >> 2) * (kKeys * 128) + (ks & 3) * 32;
              const uint32_t qoff = (ks >> 2) * (Rq * 128) + (ks & 3) * 32 + ph * (PASS == 1 ? 128 : 256) * 128;
              if (PASS == 1) {
                umma_bf16(tmem + buf * 256, umma_desc_sw128(qbase + qoff), umma_desc_sw128(kbase + koff), idesc, ks > 0);
              } else {
                umma_bf16(tmem + buf * 256, umma_desc_sw128(kbase + koff), umma_desc_sw128(qbase + qoff), idesc, ks > 0);
              }
            }
            umma_commit(&tfull[buf]);
          }
          if (!ok) break;
          umma_commit(&empty[st]);
        }
        umma_commit(qfree);
      }
      if (!ok) {
        *abort_flag = 1;
        raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
      }
      umma_commit(done);  // every MMA issued above has completed once this arrives
      mbar_wait(done, 0);
    }
  } else if (warp > kMmaWarp) {
    // ---------------- value norms: this CTA's share of the pass's rows ----------------
    // a piece takes the rows of its share of the unit's tiles, pass 1's row halves a part of them each
    int used = 0;
    for (Walk w = w0; w.left > 0; w.next(a, kKeys)) {
      const int n1 = w.n / 2;
      const int lo = PASS == 1 ? 0 : n1, hi = PASS == 1 ? n1 : w.n;
      auto edge = [&](int t) { return lo + (int)((long long)(hi - lo) * t / w.ntiles); };
      const int e0 = edge(w.t), len = edge(w.t + w.nt) - e0;
      const int parts = PASS == 1 ? MT : 1;
      const size_t row0 = (size_t)w.u * a.n_cap;
      if (!norm_rows<D, PASS, HALVES>(static_cast<const __nv_bfloat16*>(a.V) + row0 * D, a.vnorm + row0,
                              e0 + (int)((long long)len * h / parts), e0 + (int)((long long)len * (h + 1) / parts),
                              warp - kMmaWarp - 1, nring, nbar, a.flags, used))
        break;
    }
  } else {
    // ---------------- epilogue: warps 0-15 ----------------
    const int q = warp & 3, part = warp >> 2;  // lane quarter of TMEM, and which part of the work
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const float sc = a.scale_log2;
    // lane 0 waits, the warp follows its outcome (tcgen05.ld below needs the whole warp)
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      int ok = 0;
      if (lane == 0) {
        ok = !*abort_flag && mbar_wait(bar, parity);
        if (!ok && !*abort_flag) {
          *abort_flag = 1;
          raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
        }
      }
      return __shfl_sync(0xffffffffu, ok, 0) != 0;
    };
    if (PASS == 1) {
      int u = 0;  // accumulator use, as counted by the MMA thread
      for (Walk w = w0; w.left > 0; w.next(a, kKeys)) {
        const int n = w.n, t_begin = w.t, nt = w.nt;
        // this thread's query row in each half, its last visible key, and its running max (base 2,
        // scaled) and sum
        int r[HALVES], p[HALVES];
        float m_run[HALVES], l_run[HALVES];
#pragma unroll
        for (int ph = 0; ph < HALVES; ++ph) {
          r[ph] = h * kP1Rows + ph * 128 + q * 32 + lane;
          p[ph] = n - a.W + (r[ph] % a.W);
          m_run[ph] = -INFINITY;
          l_run[ph] = 0.f;
        }
        for (int t = 0; t < nt; ++t) {
          constexpr int kCols = 32 * SELKV_P1_CPW;           // this warp's keys of the tile
          const int key0 = (t_begin + t) * kKeys + part * kCols;
          const bool full_quarter = key0 + kCols - 1 <= n - a.W;  // every row sees every key of the part
#pragma unroll
          for (int ph = 0; ph < HALVES; ++ph) {
            if (ph >= nph) break;
            const int buf = u & 1;
            const bool ok = warp_wait(&tfull[buf], (u >> 1) & 1);
            ++u;
            tc_fence_after();
            // (pass 1 reads the accumulator 32 columns at a time, each load waited for before its
            // arithmetic: pipelined loads measured slower here, and leaving the max out of the chunks where
            // the last one still serves as a reference changed nothing)
            if (ok) {
#pragma unroll 1
              for (int c = 0; c < kCols; c += 32) {
                float v[32];
                tmem_ld32(tmem + lane_base + buf * 256 + part * kCols + c, v);
                float cm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                if (full_quarter) {
#pragma unroll
                  for (int i = 0; i < 32; ++i) cm[i & 3] = fmaxf(cm[i & 3], v[i]);
                } else {
#pragma unroll
                  for (int i = 0; i < 32; ++i) {
                    v[i] = key0 + c + i <= p[ph] ? v[i] : -INFINITY;
                    cm[i & 3] = fmaxf(cm[i & 3], v[i]);
                  }
                }
                // the scale is positive, so max(v) * scale is the max of the scaled logits
                const float mn = fmaxf(m_run[ph], fmaxf(fmaxf(cm[0], cm[1]), fmaxf(cm[2], cm[3])) * sc);
                if (mn != -INFINITY) {
                  const float s = rowsum32(v, sc, mn);
                  l_run[ph] = l_run[ph] * ex2_approx(m_run[ph] - mn) + s;
                  m_run[ph] = mn;
                }
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
          }
        }
        // fold the key parts of each row in part order (parts 1.. via shared memory)
        float2* st4 = reinterpret_cast<float2*>(colpart);  // [parts][128]
#pragma unroll
        for (int ph = 0; ph < HALVES; ++ph) {
          if (ph >= nph) break;
          if (ph > 0) named_bar_sync(1, kEpiWarps * 32);  // the first half's states are read
          if (part > 0) st4[part * 128 + q * 32 + lane] = make_float2(m_run[ph], l_run[ph]);
          named_bar_sync(1, kEpiWarps * 32);
          if (part == 0 && r[ph] < R) {
            float2 o[kP1Parts];
            o[0] = make_float2(m_run[ph], l_run[ph]);
#pragma unroll
            for (int k = 1; k < kP1Parts; ++k) o[k] = st4[k * 128 + q * 32 + lane];
            float M = o[0].x;
#pragma unroll
            for (int k = 1; k < kP1Parts; ++k) M = fmaxf(M, o[k].x);
            float L = 0.f;
            if (M != -INFINITY) {
#pragma unroll
              for (int k = 0; k < kP1Parts; ++k) L += o[k].y * ex2_approx(o[k].x - M);
            }
            a.rowpart[((size_t)group + w.u) * R + r[ph]] = make_float2(M, L);
          }
        }
        if (w.left > nt) named_bar_sync(1, kEpiWarps * 32);  // the next piece's states replace these
      }
    } else {
      const int klane = q * 32 + lane;   // key owned by this thread within the tile
      int u = 0;                         // accumulator use, as counted by the MMA thread
      int tt = 0;                        // tiles, over all pieces
      for (Walk w = w0; w.left > 0; w.next(a, kKeys)) {
        const int n = w.n, t_begin = w.t, nt = w.nt;
        float* attn = a.attn + (size_t)w.u * a.n_cap;
        static_assert(kEpiWarps * 32 >= 256 * HALVES, "a thread per row");
        {
          // (Q of the piece and its first tiles are on their way meanwhile)
          const int r = threadIdx.x;
          // the first unit's partials from the table: its chain of loads is not hidden by earlier tiles
          const Partials ps = w.left == w0.left ? Partials{walk.part0[group], walk.parts[group]} : partials_of(a, walk, w);
          const float x = r < R ? fold_row_tc(a, ps, r) : -INFINITY;
          if (w.left < w0.left) named_bar_sync(1, kEpiWarps * 32);  // the last piece's rows are done with
          if (r < 256 * HALVES) {
            rneg[r] = x;
            rwin[r] = r % a.W;
          }
          named_bar_sync(1, kEpiWarps * 32);
        }
        for (int t = 0; t < nt; ++t, ++tt) {
          const int key0 = (t_begin + t) * kKeys;
          const int j = key0 + klane;
          const int jrel = j - (n - a.W);  // > 0: only rows with (r mod W) >= jrel see key j
          // every key of this warp is seen by every row: the whole tile is unmasked
          const bool unmasked = key0 + q * 32 + 31 <= n - a.W;
          float acc = 0.f;
          for (int ph = 0; ph < HALVES; ++ph, ++u) {
            const int buf = u & 1;
            const bool ok = warp_wait(&tfull[buf], (u >> 1) & 1);
            tc_fence_after();
            // this part's 64 rows of the half: accumulator columns from c0, rows from r_lo
            const int c0 = part * 64, r_lo = ph * 256 + c0, r_hi = min(R, r_lo + 64);
            const uint32_t tcol = tmem + lane_base + buf * 256 + c0;
            if (ok && SELKV_P2_PIPE && r_hi - r_lo == 64 && unmasked) {
              acc += colsum64(tcol, smem_u32(rneg + r_lo), sc);
            } else if (ok) {
#pragma unroll 1
              for (int c = r_lo; c < r_hi; c += 32) {
                float v[32];
                tmem_ld32(tcol + (c - r_lo), v);
                const int cnt = min(32, r_hi - c);
                if (unmasked && cnt == 32) {
                  // sum over rows of 2^(v sc - M_r - log2(G Z_r)), pairs of rows packed; four
                  // interleaved partial sums as (0,1) and (2,3)
                  const uint64_t sc2 = pack_f2(sc, sc);
                  uint64_t a01 = pack_f2(0.f, 0.f), a23 = a01;
#pragma unroll
                  for (int i = 0; i < 32; i += 4) {
                    const float4 nm = *reinterpret_cast<const float4*>(&rneg[c + i]);  // rows c+i .. c+i+3
                    float x0, x1, x2, x3;
                    unpack_f2(ffma2(pack_f2(v[i], v[i + 1]), sc2, pack_f2(nm.x, nm.y)), x0, x1);
                    unpack_f2(ffma2(pack_f2(v[i + 2], v[i + 3]), sc2, pack_f2(nm.z, nm.w)), x2, x3);
                    a01 = fadd2(a01, pack_f2(ex2_approx(x0), ex2_approx(x1)));
                    a23 = fadd2(a23, pack_f2(ex2_approx(x2), ex2_approx(x3)));
                  }
                  float s0, s1, s2, s3;
                  unpack_f2(a01, s0, s1);
                  unpack_f2(a23, s2, s3);
                  acc += (s0 + s1) + (s2 + s3);
                } else {
                  // the end of a sequence (or rows that do not fill the chunk); the places of the rows
                  // in the window come from a table (a division per row and key made the last tile
                  // of a unit cost as much as a dozen others)
                  float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                  for (int i = 0; i < 32; ++i)
                    if (i < cnt && rwin[c + i] >= jrel) s4[i & 3] += ex2_approx(fmaf(v[i], sc, rneg[c + i]));
                  acc += (s4[0] + s4[1]) + (s4[2] + s4[3]);
                }
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
          }
          // The four row quarters' column sums of key j meet in shared memory (two buffers,
          // alternating by tile): parts 1-3 leave theirs and go on, part 0 adds them to its own in
          // quarter order and writes a_j.  A part reuses a buffer only once part 0 has read it.
          const int cb = tt & 1;
          float* cs = colpart + cb * 512;  // [4][128]
          uint64_t* cfull = &cs_full[q * 2 + cb];
          uint64_t* cempty = &cs_empty[q * 2 + cb];
          // bounded wait of every lane (each lane acquires what it then reads or overwrites)
          auto lane_wait = [&](uint64_t* bar, uint32_t parity) {
            if (*abort_flag) return;
            if (!mbar_wait(bar, parity)) {
              *abort_flag = 1;
              raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
            }
          };
          if (part > 0) {
            if (tt >= 2) lane_wait(cempty, ((tt >> 1) - 1) & 1);
            cs[part * 128 + klane] = acc;
            __syncwarp();
            if (lane == 0) mbar_arrive(cfull);
          } else {
            lane_wait(cfull, (tt >> 1) & 1);
            const float sum = ((acc + cs[128 + klane]) + cs[256 + klane]) + cs[384 + klane];
            __syncwarp();
            if (lane == 0) mbar_arrive(cempty);
            if (j < n) attn[j] = sum;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// How pass 1 cuts the tiles: row halves per CTA, splits per unit (or 0) and tiles per CTA group.
struct P1Cut {
  int halves, split, per;
};

// Shares of a pass's key tiles: `groups` CTAs (of `row_parts` each in pass 1) with the same number of
// consecutive tiles of all units, which crosses from one unit to the next; or, where it is no more tiles
// for the longest unit, every unit cut into the same number of splits, with no crossing.  A fixed grid of
// splits per unit left SMs idle where the units did not divide them (32 heads: 128 of 152 CTAs) or had
// unequal lengths (8 ragged prompts of 32k: passes 131 + 146 us, now 91 + 96; 64 of 8k: 233 + 284, now
// 195 + 221).  A crossing costs a reload of Q while the epilogue works on the two tiles in flight.
// `p1`: for pass 2, pass 1's plan.
int plan_walk(const CompressArgs& a, const SeqTable& tab, int row_parts, int keys, ScoreWalk& w, int& split, int& per,
              const P1Cut* p1 = nullptr) {
  const int groups = kPlanSMs / row_parts;
  const int units = a.B * a.Hkv;
  auto tiles = [&](int b) { return (tab.n[b] + keys - 1) / keys; };
  long long total = 0;
  int longest = 0;
  for (int b = 0; b < a.B; ++b) {
    total += (long long)tiles(b) * a.Hkv;
    longest = tiles(b) > longest ? tiles(b) : longest;
  }
  per = (int)((total + groups - 1) / groups);
  split = units <= groups ? groups / units : 0;
  if (split > longest) split = longest;
  if (split > 0 && (longest + split - 1) / split > per) split = 0;
  int used = 0;
  if (split > 0) {
    for (int u = 0; u < units; ++u) {
      const int T = tiles(u / a.Hkv), p = (T + split - 1) / split;
      for (int k = 0; k < split; ++k, ++used) {
        w.u0[used] = u;
        w.t0[used] = k * p;
        w.cnt[used] = T - k * p < p ? (T - k * p > 0 ? T - k * p : 0) : p;
      }
    }
  } else {
    int b = 0;
    long long before = 0;  // tiles of the sequences before b
    for (long long g = 0; g < total; g += per, ++used) {
      while (g >= before + (long long)tiles(b) * a.Hkv) before += (long long)tiles(b++) * a.Hkv;
      const int T = tiles(b), in = (int)(g - before);
      w.u0[used] = b * a.Hkv + in / T;
      w.t0[used] = in % T;
      w.cnt[used] = (int)(total - g < per ? total - g : per);
    }
  }
  for (int c = 0; c < used; ++c) {
    const int b = w.u0[c] / a.Hkv;
    w.n[c] = tab.n[b];
    if (p1 == nullptr) continue;
    const int T1 = score_tc_tiles1(tab.n[b]);
    const Partials ps = partials_of(p1->split, p1->per, w.u0[c], tab.t1[b] * a.Hkv + w.u0[c] % a.Hkv * T1, T1);
    w.part0[c] = ps.first;
    w.parts[c] = ps.count;
  }
  return used;
}

// Row halves of a CTA in pass 1.  Two 128-row halves read a tile's keys once for both, where two CTAs with
// a half each read them twice (from L2, or HBM where they drift apart: 8 x 32k 100 -> 90 us, 64 x 8k
// 215 -> 197); but a CTA's share is then twice as coarse.  From 8 tiles (16 accumulators) a CTA on, unless
// rounding to whole tiles makes it longer (16k: 8 accumulators against 7, 18.9 against 16.4 us).
int p1_halves(const CompressArgs& a, const SeqTable& tab) {
  long long total = 0;
  for (int b = 0; b < a.B; ++b) total += (long long)score_tc_tiles1(tab.n[b]) * a.Hkv;
  auto accs = [&](int halves) {  // accumulators of the longest share
    const int groups = kPlanSMs / ((a.R + 128 * halves - 1) / (128 * halves));
    return (total + groups - 1) / groups * halves;
  };
  return a.R > 128 && accs(2) >= 16 && accs(2) <= accs(1) ? 2 : 1;
}
int p1_row_parts(int R, int halves) { return (R + 128 * halves - 1) / (128 * halves); }

// Both passes' shares: the CTA groups of pass 1 and the CTAs of pass 2.
void plan_passes(const CompressArgs& a, const SeqTable& tab, ScoreWalk& w1, ScoreWalk& w2, P1Cut& cut, int& groups1,
                 int& groups2) {
  cut.halves = p1_halves(a, tab);
  groups1 = plan_walk(a, tab, p1_row_parts(a.R, cut.halves), SELKV_P1_KEYS, w1, cut.split, cut.per);
  int split2, per2;
  groups2 = plan_walk(a, tab, 1, kP2Keys, w2, split2, per2, &cut);
  w2.p1_split = cut.split;
  w2.p1_per = cut.per;
}

template <int D, int H1, int H2>
cudaError_t launch_tc_t(const CompressArgs& a, const ScoreWalk& w1, const ScoreWalk& w2, int groups1, int groups2,
                        cudaStream_t st, int passes) {
  using C1 = SCfg<D, 1, H1>;
  using C2 = SCfg<D, 2, H2>;
  CUtensorMap tq, tk1, tk2;
  if (!encode_rows_bf16(&tq, a.Q, (uint64_t)a.B * a.Hq * a.W, D, 128) ||
      !encode_rows_bf16(&tk1, a.K, (uint64_t)a.B * a.Hkv * a.n_cap, D, C1::kKeys) ||
      !encode_rows_bf16(&tk2, a.K, (uint64_t)a.B * a.Hkv * a.n_cap, D, C2::kKeys))
    return cudaErrorInvalidValue;
  if (passes & kScoreRowstats) {
    cudaError_t e = set_smem_once<score_tc_kernel<D, 1, H1>>(C1::kSmem);
    if (e != cudaSuccess) return e;
    launch_chained(a.chain, score_tc_kernel<D, 1, H1>, groups1 * p1_row_parts(a.R, H1), cta_threads(1, H1, a.V != nullptr),
                   C1::kSmem, st, tq, tk1, a, w1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (!(passes & kScoreColsums)) return cudaSuccess;
  if (passes & kScoreRowstats) {
    const cudaError_t e = set_smem_once<score_tc_kernel<D, 2, H2>>(C2::kSmem);
    if (e != cudaSuccess) return e;
    launch_chained(a.chain, score_tc_kernel<D, 2, H2>, groups2, cta_threads(2, H2, a.V != nullptr), C2::kSmem, st, tq, tk2,
                   a, w2);
  } else {  // (alone, it follows a kernel of the caller's and starts only after it)
    const cudaError_t e = set_smem_once<score_tc_kernel<D, 2, H2, true>>(C2::kSmem);
    if (e != cudaSuccess) return e;
    launch_chained(false, score_tc_kernel<D, 2, H2, true>, kPlanSMs, cta_threads(2, H2, a.V != nullptr), C2::kSmem, st, tq,
                   tk2, a, w2);
  }
  return cudaGetLastError();
}

}  // namespace

// The window rows of a KV group, R = G W, go to the tensor cores up to 512 (two 256-row halves
// in the column-sum pass); wider groups take the CUDA-core path.
bool score_uses_tc(int dtype, int D, int R) { return dtype == SELKV_BF16 && (D == 64 || D == 128) && R >= 1 && R <= 512; }

// Row-statistics partials of pass 1: one per CTA group and unit it holds tiles of, at (group + unit),
// which is another for every such pair (both only grow along the list of tiles).
size_t score_tc_partials(int B, int Hkv) { return (size_t)B * Hkv + kPlanSMs; }

int score_tc_tiles1(int n) { return (n + SELKV_P1_KEYS - 1) / SELKV_P1_KEYS; }

ScoreWalk plan_colsums(const CompressArgs& a, const SeqTable& tab) {
  ScoreWalk w1{}, w2{};
  P1Cut cut;
  int groups1, groups2;
  plan_passes(a, tab, w1, w2, cut, groups1, groups2);
  return w2;
}

cudaError_t launch_score_tc(const CompressArgs& a, const SeqTable& tab, cudaStream_t st, int passes) {
  ScoreWalk w1{}, w2{};
  P1Cut cut;
  int groups1, groups2;
  plan_passes(a, tab, w1, w2, cut, groups1, groups2);
  auto go = [&](auto d, auto h2) {
    constexpr int D = decltype(d)::value, H2 = decltype(h2)::value;
    return cut.halves == 2 ? launch_tc_t<D, 2, H2>(a, w1, w2, groups1, groups2, st, passes)
                           : launch_tc_t<D, 1, H2>(a, w1, w2, groups1, groups2, st, passes);
  };
  using std::integral_constant;
  if (a.R > 256) return a.D == 128 ? go(integral_constant<int, 128>{}, integral_constant<int, 2>{}) : go(integral_constant<int, 64>{}, integral_constant<int, 2>{});
  return a.D == 128 ? go(integral_constant<int, 128>{}, integral_constant<int, 1>{}) : go(integral_constant<int, 64>{}, integral_constant<int, 1>{});
}

}  // namespace selkv
