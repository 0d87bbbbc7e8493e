// Routing, gated merge and kept-row copy in one kernel, for bf16 caches with 32-token buckets.
//
// The same results as route_kernel and merge_kernel of merge.cu (Eq. 3-6 with the nearest-ring
// rule for empty buckets).  A bucket is then one word of the selection's kept mask, one lane per
// token, and an 8 KB tile (d = 128) of value rows:
//   * a one-warp CTA walks `seg` consecutive buckets of a (sequence, KV head) as targets X and
//     streams the value tiles of every bucket whose tokens route to them (a contiguous range:
//     each empty bucket belongs to one neighbour) through a two-stage ring of TMA loads;
//   * tau_X is an argmax over the lanes; the next non-empty bucket R is found in the mask words
//     and its `a` values, which decide the ties of the empty buckets between, are then X's when R's
//     turn comes;
//   * the cosines of a bucket's 32 tokens with v_tau are one small tensor-core product (tokens x d
//     times d x 8, every column v_tau): bf16 products are exact and the sums fp32;
//   * sum_j w_j v_j is another (d x tokens times tokens x 8): column 0 holds the weights' upper 8
//     bits, columns 1 and 2 the next two 8, so together all 24 bits of the fp32 weights count;
//   * the kept value rows are copied from the tile; the kept key rows by other warps of the same launch,
//     64 slots each, with bulk copies in and out of shared memory.
// A bucket takes about 450 warp instructions where the CUDA-core kernel took 1900 (unpacking,
// shuffles, one row at a time) and lane 0 keeps 16 KB per warp in flight without registers.
// It is bound by HBM on long sequences: one layer of 8 x 100k rows at 25% (358 MB) takes 67 us, 64 x
// 8k at 10% (1.04 GB) 182 us, 80% and 84% of the copy rate (83 and 275 us before, with 9 and 15 us of
// route kernel on top); short ones by a walk's chain of dependent loads.
#include <climits>

#include "ptx.cuh"
#include "rope.cuh"
#include "selkv_internal.cuh"

namespace selkv {
namespace {

constexpr int kStages = 2;       // value tiles in flight per warp
constexpr int kCtasPerSm = 12;   // one-warp CTAs resident per SM (18 KB of shared memory each)
constexpr int kKeySlots = 64;    // key rows a copying warp moves
#ifndef SELKV_MERGE_SEG
#define SELKV_MERGE_SEG 8  // most buckets a warp walks
#endif
constexpr uint32_t kFull = 0xffffffffu;
// The weights go to the product times 2^40, so that the lower pieces of the smallest ones are not lost
// among bf16's subnormals (a weight of 2^-125 kept 9 of its 24 bits).  A power of two changes no other
// result.  The weights of a target add up to at most W, and the elements of a row with a finite norm are
// below 2^64, so nothing overflows for W up to 2^24.
constexpr float kWeightUp = 0x1p40f, kWeightDown = 0x1p-40f;

template <int D>
struct MCfg {
  static constexpr int kBoxes = D / 64;
  static constexpr int kBoxBytes = 32 * 128;
  static constexpr int kTileBytes = kBoxes * kBoxBytes;
  static constexpr int kWLd = 80;  // bytes per weight row (32 bf16, padded against bank conflicts)
  // ring | v_tau (D bf16) | weights [8][kWLd] | weighted sum (D floats) | kept lanes [32] | barriers
  static constexpr int kVt = kStages * kTileBytes;
  static constexpr int kW = kVt + D * 2;
  static constexpr int kNum = kW + 8 * kWLd;
  static constexpr int kList = kNum + D * 4;
  static constexpr int kBars = kList + 32;
  static constexpr int kSmem = kBars + kStages * 8;
  static_assert(kVt % 1024 == 0 && kW % 16 == 0 && kNum % 16 == 0 && kBars % 8 == 0, "alignment");
};

// The kept masks of 32 consecutive buckets (one per lane), moved along as the walk asks for more.
struct MaskWindow {
  const uint2* km;
  int nb, base, lane;
  uint2 w;
  uint32_t any;
  __device__ __forceinline__ void load(int from) {
    base = from;
    w = from + lane < nb ? km[from + lane] : make_uint2(0u, 0u);
    any = __ballot_sync(kFull, w.x != 0u);
  }
  // First non-empty bucket at or after `from` (nb: none), inside the window afterwards.
  __device__ __forceinline__ int next(int from) {
    while (from < nb) {
      if (from >= base + 32) load(from);
      const uint32_t bits = any >> (from - base);
      if (bits) return from + __ffs(bits) - 1;
      from = base + 32;
    }
    return nb;
  }
  __device__ __forceinline__ uint32_t mask(int e) const { return __shfl_sync(kFull, w.x, e - base); }
  __device__ __forceinline__ int slot0(int e) const { return (int)__shfl_sync(kFull, w.y, e - base); }
};

// Lane of the kept token with the largest a, ties to the lower position; `best` gets its a.  a is
// never negative, so its bits order as the values do.
__device__ __forceinline__ int argmax_kept(uint32_t mask, float a, int lane, float& best) {
  const uint32_t key = (mask >> lane) & 1u ? __float_as_uint(a) : 0u;
  const uint32_t mx = __reduce_max_sync(kFull, key);
  best = __uint_as_float(mx);
  return __ffs(__ballot_sync(kFull, ((mask >> lane) & 1u) && key == mx)) - 1;
}

// Turn the staged key rows back by e w_f, e = position - slot: a lane takes the pairs of two
// frequencies of a row.
template <int D>
__device__ __forceinline__ void turn_rows(const CompressArgs& a, const int (&pos)[kKeySlots / 32], int s0, int rows,
                                          unsigned char* ring) {
  constexpr int LP = D / 4, RPI = 32 / LP;  // lanes per row, rows per step
  const int sub = (int)threadIdx.x / LP, f0 = (int)threadIdx.x % LP * 2;
  // HALF pairs (f, f + d/2), INTERLEAVED (2 f, 2 f + 1)
  const bool half = a.rope == SELKV_ROPE_HALF;
  const int o0 = half ? f0 : 2 * f0, o1 = half ? f0 + D / 2 : 2 * f0 + 2;  // this lane's two 4-byte words
#pragma unroll
  for (int i = 0; i < kKeySlots / 32; ++i) {
#pragma unroll 4
    for (int k = 0; k < 32; k += RPI) {
      const int r = i * 32 + k + sub;
      const int e = max(0, __shfl_sync(kFull, pos[i], k + sub) - (s0 + r));  // kept positions ascend with their slots
      if (r >= rows) continue;
      uint32_t* w0 = reinterpret_cast<uint32_t*>(ring + (r * D + o0) * 2);
      uint32_t* w1 = reinterpret_cast<uint32_t*>(ring + (r * D + o1) * 2);
      const uint32_t u0 = *w0, u1 = *w1;
      float x0 = bf16_lo(u0), x1 = bf16_hi(u0), y0 = bf16_lo(u1), y1 = bf16_hi(u1);
      float2 cs[2];
      rope_angles<2>(a, f0, e, cs);
      if (half) {
        rope_back(x0, y0, cs[0]);
        rope_back(x1, y1, cs[1]);
      } else {
        rope_back(x0, x1, cs[0]);
        rope_back(y0, y1, cs[1]);
      }
      *w0 = pack_bf16(x0, x1);
      *w1 = pack_bf16(y0, y1);
    }
  }
}

// Key rows of slots [s0, s0 + kKeySlots) of (sequence, KV head) bk, a warp's work: one bulk copy a row
// into the idle ring, then all of them to the slots, which are consecutive, with one; in between, with
// repositioning, each is turned by the shift from its position to its slot.
template <int D>
__device__ __forceinline__ void copy_keys(const CompressArgs& a, int bk, size_t unit, int s0, int m, unsigned char* ring,
                                          uint64_t* bar) {
  static_assert(kKeySlots * D * 2 <= MCfg<D>::kVt && kKeySlots % 32 == 0, "the ring holds the rows");
  const int lane = threadIdx.x, rows = min(kKeySlots, m - s0);
  if (rows <= 0) return;
  const __nv_bfloat16* Kb = static_cast<const __nv_bfloat16*>(a.K) + (size_t)bk * a.n_cap * D;
  int pos[kKeySlots / 32];
  bool in = true;
#pragma unroll
  for (int i = 0; i < kKeySlots / 32; ++i) {
    const int r = i * 32 + lane;
    pos[i] = r < rows ? a.kept_pos[unit * a.m_cap + s0 + r] : 0;
    in = in && pos[i] >= 0 && pos[i] < a.n_cap;
  }
  if (!__all_sync(kFull, in)) {  // (cannot happen: the selection writes them)
    if (lane == 0) raise_flag(a.flags, SELKV_DEVERR_COUNT);
    return;
  }
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar, (uint32_t)rows * D * 2);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kKeySlots / 32; ++i) {
    const int r = i * 32 + lane;
    if (r < rows) bulk_load(ring + r * D * 2, Kb + (size_t)pos[i] * D, D * 2, bar);
  }
  if (!__all_sync(kFull, mbar_wait(bar, 0))) {
    if (lane == 0) raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
    mbar_wait(bar, 0);  // (bounded) the copies land before the CTA leaves
    return;
  }
  if (a.rope != SELKV_ROPE_OFF) {
    turn_rows<D>(a, pos, s0, rows, ring);
    fence_proxy_async_smem();  // the turned rows, before the bulk copy reads them
    __syncwarp();
  }
  if (lane == 0) {
    bulk_store(static_cast<__nv_bfloat16*>(a.Kc) + ((size_t)bk * a.m_cap + s0) * D, ring, (uint32_t)rows * D * 2);
    bulk_store_wait();
  }
}

template <int D>
__global__ __launch_bounds__(32, kCtasPerSm) void merge_mma_kernel(const __grid_constant__ CUtensorMap tmV,
                                                                  CompressArgs a, int seg, int walks) {
  chain_begin();
  using C = MCfg<D>;
  using bf16 = __nv_bfloat16;
  constexpr int PER = D / 32;        // elements of a row per lane
  constexpr int LPR = D / 8;         // lanes per row at 16 bytes a lane
  constexpr int RPI = 32 / LPR;      // rows per warp load
  constexpr int MT = D / 16, KS = D / 16;
  extern __shared__ __align__(1024) unsigned char smem[];
  float* nums = reinterpret_cast<float*>(smem + C::kNum);
  unsigned char* list = smem + C::kList;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kBars);
  const int lane = threadIdx.x;
  const int bk = blockIdx.y, b = bk / a.Hkv, kv = bk % a.Hkv;
  if ((int)blockIdx.x >= walks) {
    copy_keys<D>(a, bk, sel_unit(a, b, kv), ((int)blockIdx.x - walks) * kKeySlots, a.seq_m[b], smem, bars);
    return;
  }
  const int n = a.seq_n[b], nb = (n + 31) / 32;
  const int x0 = blockIdx.x * seg, x1 = min(nb, x0 + seg);
  if (x0 >= nb) return;
  const size_t row_base = (size_t)bk * a.n_cap;
  const float* A = a.attn + row_base;
  const float* vn = a.vnorm + row_base;
  const bool expand = a.empty_bucket == SELKV_EMPTY_EXPAND;
  MaskWindow win{a.kmask + sel_unit(a, b, kv) * a.kmask_ld, nb, x0, lane, make_uint2(0u, 0u), 0u};
  win.load(x0);

  // Last non-empty bucket before x0 (-1: none) and its mask.
  int L = -1;
  uint32_t maskL = 0u;
  if (expand)
    for (int e0 = x0 - 1; e0 >= 0 && L < 0; e0 -= 32) {
      const uint32_t w = e0 - lane >= 0 ? win.km[e0 - lane].x : 0u;
      const uint32_t any = __ballot_sync(kFull, w != 0u);
      if (any) {
        L = e0 - (__ffs(any) - 1);
        maskL = __shfl_sync(kFull, w, __ffs(any) - 1);
      }
    }

  auto dbg_untargeted = [&](int from, int to) {  // empty buckets whose tokens have no target
    if (a.dbg_target == nullptr && a.dbg_gate == nullptr && a.dbg_decision == nullptr) return;
    for (int j = from * 32 + lane; j < min(n, to * 32); j += 32) {
      if (a.dbg_target) a.dbg_target[row_base + j] = -1;
      if (a.dbg_gate) a.dbg_gate[row_base + j] = 0.f;
      if (a.dbg_decision) a.dbg_decision[row_base + j] = 0;
    }
  };
  int X = win.next(x0);
  if (!expand || a.seq_m[b] == 0) dbg_untargeted(x0, min(X, x1));
  if (X >= x1) return;

  if (lane < kStages) mbar_init(&bars[lane], 1);
  for (int i = lane; i < 8 * C::kWLd / 4; i += 32) reinterpret_cast<uint32_t*>(smem + C::kW)[i] = 0u;
  fence_mbar_init();
  __syncwarp();

  // Tiles are issued and consumed in ascending bucket order; `next_e` is the next one to issue.
  int issued = 0, consumed = 0, next_e = 0;
  auto issue = [&](int e) {
    if (lane == 0) {
      const int st = issued % kStages;
      mbar_arrive_expect_tx(&bars[st], C::kTileBytes);
#pragma unroll
      for (int bx = 0; bx < C::kBoxes; ++bx)
        tma_load_2d(smem + st * C::kTileBytes + bx * C::kBoxBytes, &tmV, bx * 64, (int)row_base + e * 32, &bars[st]);
    }
    ++issued;
    next_e = e + 1;
  };
  auto wait_tile = [&]() -> bool {
    return __all_sync(kFull, mbar_wait(&bars[consumed % kStages], (consumed / kStages) & 1));
  };
  auto prefetch = [&]() {
    while (next_e < x1 && issued - consumed < kStages) issue(next_e);
  };

  const int mi = lane >> 3, ri = lane & 7, g8 = lane >> 2, c4 = lane & 3;
  const bf16* Vb = static_cast<const bf16*>(a.V) + row_base * D;
  bf16* Vc = static_cast<bf16*>(a.Vc) + (size_t)bk * a.m_cap * D;

  uint32_t mask = win.mask(X);
  int slot0 = win.slot0(X);
  float AX = X * 32 + lane < n ? A[X * 32 + lane] : 0.f;
  float NX = X * 32 + lane < n ? vn[X * 32 + lane] : 0.f;
  float a_tau;
  int tl = argmax_kept(mask, AX, lane, a_tau);  // tau = 32 X + tl
  // First bucket that routes to X.  An empty e between L and X goes to the nearer one; at equal
  // distance both are in the ring and X wins only with a strictly larger a (tau_L has the lower
  // index).  Towards R, X wins ties at equal distance (tau_X has the lower index).
  int lo = X;
  if (expand) {
    if (L < 0) {
      lo = 0;
    } else if (L < X - 1) {
      lo = (X + L) / 2 + 1;
      if (((X + L) & 1) == 0) {
        float aL;
        argmax_kept(maskL, A[L * 32 + lane], lane, aL);
        if (a_tau > aL) lo = (X + L) / 2;
      }
    }
  }
  next_e = lo;
  issue(lo);
  prefetch();

  // What the next target needs is loaded a target ahead: its a and norms, and v_tau of it as soon as
  // its a decide tau.
  RowSlice<bf16, PER> vt;
  vt.load(Vb + ((size_t)X * 32 + tl) * D + lane * PER);
  uint32_t maskR = 0u;
  int slotR = 0;
  float AR = 0.f, NR = 0.f;
  auto fetch = [&](int e) {
    maskR = win.mask(e);
    slotR = win.slot0(e);
    const int j = e * 32 + lane;
    AR = j < n ? A[j] : 0.f;
    NR = j < n ? vn[j] : 0.f;
  };
  int R = win.next(X + 1);
  if (R < nb) fetch(R);

  bool ok = true;
  while (true) {
    bf16* vts = reinterpret_cast<bf16*>(smem + C::kVt);
    const float vn_tau = __shfl_sync(kFull, NX, tl);
    int hi = X;
    const uint32_t below = mask & ((1u << lane) - 1u);
    const bool keptX = (mask >> lane) & 1u;
    const int nk = __popc(mask);
    if (keptX) list[__popc(below)] = (unsigned char)lane;
    if (lane * PER < D) {
      if constexpr (PER == 4) *reinterpret_cast<uint2*>(vts + lane * PER) = vt.w;
      else *reinterpret_cast<uint32_t*>(vts + lane * PER) = vt.w;
    }
    __syncwarp();
    const int sub = lane / LPR, sl = lane % LPR;
    uint32_t vb[2 * KS];  // B fragments of v_tau, every column the same
#pragma unroll
    for (int i = 0; i < KS / 2; ++i) {
      uint32_t f[4];
      ldmatrix_x4(f, smem_u32(vts) + (i * 4 + mi) * 16);
#pragma unroll
      for (int t = 0; t < 4; ++t) vb[4 * i + t] = f[t];
    }
    // the next target's tau, and with its a the last bucket that routes to X
    const int Y = R;  // the next target (nb: none)
    const uint32_t maskY = maskR;
    const int slotY = slotR;
    const float AY = AR, NY = NR;
    float aY = 0.f;
    int tY = 0;
    RowSlice<bf16, PER> vtY;
    vtY.zero();
    if (Y < nb) {
      tY = argmax_kept(maskY, AY, lane, aY);
      if (Y < x1) {
        vtY.load(Vb + ((size_t)Y * 32 + tY) * D + lane * PER);
        R = win.next(Y + 1);
        if (R < nb) fetch(R);
      }
    }
    if (expand) {
      if (Y >= nb) {
        hi = nb - 1;
      } else if (Y > X + 1) {
        hi = (X + Y - 1) / 2;
        if (((X + Y) & 1) == 0 && a_tau >= aY) hi = (X + Y) / 2;
      }
    }
    if (nk > 0 && (slot0 < 0 || slot0 + nk > a.m_cap)) {  // (cannot happen: the selection keeps m <= m_cap)
      if (lane == 0) raise_flag(a.flags, SELKV_DEVERR_COUNT);
      break;
    }

    float acc[MT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][e] = 0.f;
    float extra[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) extra[t] = 0.f;
    float den = 0.f;
    int merged = 0;  // contributors with g > 0 (the count bias)
    for (int e = lo; e <= hi; ++e) {
      const int base = e * 32, cnt = min(32, n - base);
      const bool in = lane < cnt;
      const float Ae = e == X ? AX : (in ? A[base + lane] : 0.f);
      const float Ne = e == X ? NX : (in ? vn[base + lane] : 0.f);
      const bool con = in && !(e == X && keptX);  // this lane's token is merged (or dropped) here
      if (next_e <= e) issue(e);
      if (!wait_tile()) {
        ok = false;
        break;
      }
      unsigned char* tile = smem + (consumed % kStages) * C::kTileBytes;
      const uint32_t T = smem_u32(tile);
      if (e == X) {
        // the kept rows but the target's, from the tile to their slots
        for (int r = sub; r < nk; r += RPI) {
          const int row = list[r];
          const uint4 v = *reinterpret_cast<const uint4*>(tile + (sl >> 3) * C::kBoxBytes + swz128(row, sl & 7));
          if (row != tl) *reinterpret_cast<uint4*>(Vc + (size_t)(slot0 + r) * D + sl * 8) = v;
        }
      }
      float g = a.gate_mode == SELKV_GATE_OPEN ? 1.f : 0.f;
      if (a.gate_mode == SELKV_GATE_COSINE) {
        float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const int chunk = ks * 2 + (mi >> 1);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t f[4];
            ldmatrix_x4(f, T + (chunk >> 3) * C::kBoxBytes + swz128(h * 16 + (mi & 1) * 8 + ri, chunk & 7));
            mma_bf16_16816(d[h], f, vb[2 * ks], vb[2 * ks + 1]);
          }
        }
        // lane (g8, c4) holds tokens g8, 8 + g8, 16 + g8, 24 + g8 in every column: hand each its own
        const float pick = c4 == 0 ? d[0][0] : c4 == 1 ? d[0][2] : c4 == 2 ? d[1][0] : d[1][2];
        const float dot = __shfl_sync(kFull, pick, (lane & 7) * 4 + (lane >> 3));
        const float sim = (Ne == 0.f || vn_tau == 0.f) ? 0.f : dot / (Ne * vn_tau);
        g = fminf(fmaxf(sim, 0.f), 1.f);
      }
      const float w = con ? g * Ae : 0.f;
      den += w;
      merged += __popc(__ballot_sync(kFull, con && g > 0.f));
      if (con) {
        const size_t o = row_base + base + lane;
        if (a.dbg_target) a.dbg_target[o] = X * 32 + tl;
        if (a.dbg_gate) a.dbg_gate[o] = g;
        if (a.dbg_decision) a.dbg_decision[o] = g > 0.f ? 1 : 0;
      }
      // the weight in three bf16 pieces
      const float ws = w * kWeightUp;
      const bf16 w0 = __float2bfloat16_rn(ws);
      const float r1 = ws - __bfloat162float(w0);
      const bf16 w1 = __float2bfloat16_rn(r1);
      const bf16 w2 = __float2bfloat16_rn(r1 - __bfloat162float(w1));
      bf16* wrow = reinterpret_cast<bf16*>(smem + C::kW) + lane;
      wrow[0] = w0;
      wrow[C::kWLd / 2] = w1;
      wrow[C::kWLd] = w2;
      // Rows that do not contribute have weight 0, but 0 times inf or NaN would still reach the
      // sum: rows past n, and rows whose norm is not finite, are cleared first.  Of the latter the
      // contributors are added here (a piece of a weight may be 0 where the weight is not).
      uint32_t bad = __ballot_sync(kFull, !in || !(Ne < INFINITY));
      const uint32_t cons = __ballot_sync(kFull, con);
      const bool cleared = bad != 0u;
      if (cleared) __syncwarp();  // other lanes' reads of these rows (the copy of the kept ones, the cosines) come first
      for (; bad; bad &= bad - 1u) {
        const int row = __ffs(bad) - 1;
        if ((cons >> row) & 1u) {
          const float wr = __shfl_sync(kFull, w, row);
          const int d0 = lane * PER;
          const bf16* src = reinterpret_cast<const bf16*>(tile + (d0 / 64) * C::kBoxBytes + swz128(row, (d0 % 64) / 8)) + d0 % 8;
#pragma unroll
          for (int t = 0; t < PER; ++t) extra[t] = fmaf(wr, __bfloat162float(src[t]), extra[t]);
          __syncwarp();
        }
        if (lane < LPR)
          *reinterpret_cast<uint4*>(tile + (lane >> 3) * C::kBoxBytes + row * 128 + (lane & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
      }
      __syncwarp();
      uint32_t wb[4];  // B fragments: row n of the weights is column n
      ldmatrix_x4(wb, smem_u32(smem + C::kW) + ri * C::kWLd + mi * 16);
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int chunk = m * 2 + (mi & 1);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint32_t f[4];
          ldmatrix_x4_trans(f, T + (chunk >> 3) * C::kBoxBytes + swz128(ks * 16 + (mi >> 1) * 8 + ri, chunk & 7));
          mma_bf16_16816(acc[m], f, wb[2 * ks], wb[2 * ks + 1]);
        }
      }
      if (cleared) fence_proxy_async_smem();  // before the stage is loaded again
      __syncwarp();
      ++consumed;
      prefetch();
    }
    if (!ok) break;

    // the target's value row: columns 0-2 of the product added up, a row's elements to its lane
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      float s0 = acc[m][0] + acc[m][1], s1 = acc[m][2] + acc[m][3];
      s0 += __shfl_xor_sync(kFull, s0, 1);
      s1 += __shfl_xor_sync(kFull, s1, 1);
      if (c4 == 0) {
        nums[m * 16 + g8] = s0 * kWeightDown;
        nums[m * 16 + 8 + g8] = s1 * kWeightDown;
      }
    }
    den = warp_sum(den);
    __syncwarp();
    const float tot = a_tau + den;
    bf16* dst = Vc + (size_t)(slot0 + __popc(mask & ((1u << tl) - 1u))) * D + lane * PER;
    float vm[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) vm[t] = tot > 0.f ? (a_tau * vt[t] + (nums[lane * PER + t] + extra[t])) / tot : vt[t];
    if constexpr (PER == 4) store4(dst, vm);
    else *reinterpret_cast<uint32_t*>(dst) = pack_bf16(vm[0], vm[1]);
    if (keptX) {
      const size_t s = (size_t)bk * a.m_cap + slot0 + __popc(below);
      const float ratio = lane == tl && a_tau > 0.f ? tot / a_tau : 1.f;
      const float count = lane == tl ? (float)merged : 0.f;
      a.ratio[s] = ratio;
      a.mcount[s] = count;
      if (a.dbg_ratio) a.dbg_ratio[s] = ratio;
      const size_t o = row_base + X * 32 + lane;
      if (a.dbg_target) a.dbg_target[o] = -1;
      if (a.dbg_gate) a.dbg_gate[o] = 0.f;
      if (a.dbg_decision) a.dbg_decision[o] = 2;
    }
    __syncwarp();  // the lists and sums are read; the next target rewrites them

    if (!expand) {
      dbg_untargeted(X + 1, min(Y, x1));
      if (Y < x1) {  // step over the tiles of the empty buckets between
        for (int e = X + 1; e < Y && ok; ++e)
          if (e < next_e) {
            ok = wait_tile();
            ++consumed;
          }
        next_e = max(next_e, Y);
      }
    }
    if (Y >= x1 || !ok) break;
    X = Y;
    mask = maskY;
    slot0 = slotY;
    AX = AY;
    NX = NY;
    tl = tY;
    a_tau = aY;
    vt = vtY;
    lo = expand ? hi + 1 : X;
  }
  if (!ok && lane == 0) raise_flag(a.flags, SELKV_DEVERR_TIMEOUT);
  for (; consumed < issued; ++consumed) wait_tile();  // (bounded) tiles in flight land before the CTA leaves
}

template <int D>
cudaError_t launch_t(const CompressArgs& a, cudaStream_t s) {
  CUtensorMap tv;
  if (!encode_rows_bf16(&tv, a.V, (uint64_t)a.B * a.Hkv * a.n_cap, D, 32)) return cudaErrorInvalidValue;
  const cudaError_t e = set_smem_once<merge_mma_kernel<D>>(MCfg<D>::kSmem);
  if (e != cudaSuccess) return e;
  // Buckets per warp: up to 8 (a walk starts with two dependent rounds of loads), fewer where the
  // warps would not fill the SMs: one and a half times what would fill them with walks alone, which
  // leaves room for the key warps in the same wave (8 heads x 16k: 3 buckets 18 us, 2 or 4 21).
  const int units = a.B * a.Hkv, nb = (a.n_cap + 31) / 32;
  const long long per = (long long)units * nb * 3 / (2 * kPlanSMs * kCtasPerSm);
  const int seg = (int)(per < 1 ? 1 : per > SELKV_MERGE_SEG ? SELKV_MERGE_SEG : per);
  const int walks = (nb + seg - 1) / seg;
  const int keys = (a.m_cap + kKeySlots - 1) / kKeySlots;
  launch_chained(a.chain, merge_mma_kernel<D>, dim3(walks + keys, units), 32, MCfg<D>::kSmem, s, tv, a, seg, walks);
  return cudaGetLastError();
}

}  // namespace

bool merge_uses_mma(int dtype, int D, int bucket, int routing) {
  return dtype == SELKV_BF16 && (D == 64 || D == 128) && bucket == 32 && routing == SELKV_ROUTE_BUCKET;
}

cudaError_t launch_merge_mma(const CompressArgs& a, cudaStream_t s) {
  return a.D == 128 ? launch_t<128>(a, s) : launch_t<64>(a, s);
}

}  // namespace selkv
