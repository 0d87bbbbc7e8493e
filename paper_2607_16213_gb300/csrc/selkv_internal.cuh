// Internal declarations shared by the SelKV kernels and the C-ABI host code.
#pragma once

#include <atomic>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/selkv.h"

namespace selkv {

// Every workspace starts with this header; the rest is carved by the host planners.
struct WsHeader {
  uint32_t flags;  // SELKV_DEVERR_* bits, sticky until selkv_workspace_error
  uint32_t pad[63];
};
static_assert(sizeof(WsHeader) == 256, "header is 256 bytes");

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void raise_flag(uint32_t* flags, uint32_t bit) { atomicOr(flags, bit); }

// ---- element access: storage dtype -> fp32 ------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Load 8 consecutive elements starting at p (16-byte aligned for bf16, 32-byte for fp32).
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  x[0] = bf16_lo(u.x); x[1] = bf16_hi(u.x);
  x[2] = bf16_lo(u.y); x[3] = bf16_hi(u.y);
  x[4] = bf16_lo(u.z); x[5] = bf16_hi(u.z);
  x[6] = bf16_lo(u.w); x[7] = bf16_hi(u.w);
}
__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0];
  const float4 b = reinterpret_cast<const float4*>(p)[1];
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
  x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
// Load 4 consecutive elements (8-byte aligned for bf16, 16-byte for fp32).
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&x)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  x[0] = bf16_lo(u.x); x[1] = bf16_hi(u.x);
  x[2] = bf16_lo(u.y); x[3] = bf16_hi(u.y);
}
__device__ __forceinline__ void load4(const float* p, float (&x)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
}
__device__ __forceinline__ void load2(const __nv_bfloat16* p, float (&x)[2]) {
  const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
  x[0] = bf16_lo(u); x[1] = bf16_hi(u);
}
__device__ __forceinline__ void load2(const float* p, float (&x)[2]) {
  const float2 a = *reinterpret_cast<const float2*>(p);
  x[0] = a.x; x[1] = a.y;
}
__device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float load1(const float* p) { return *p; }

__device__ __forceinline__ void store1(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void store1(float* p, float v) { *p = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float (&x)[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(x[0], x[1]);
  __nv_bfloat162 b = __floats2bfloat162_rn(x[2], x[3]);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}
__device__ __forceinline__ void store4(float* p, const float (&x)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
}

// One lane's PER consecutive elements of a row, kept in the storage type.
template <typename T, int PER>
struct RowSlice;
template <>
struct RowSlice<__nv_bfloat16, 4> {
  uint2 w;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { w = *reinterpret_cast<const uint2*>(p); }
  __device__ __forceinline__ void zero() { w = make_uint2(0u, 0u); }
  __device__ __forceinline__ float operator[](int e) const {
    const uint32_t x = e < 2 ? w.x : w.y;
    return (e & 1) ? bf16_hi(x) : bf16_lo(x);
  }
};
template <>
struct RowSlice<__nv_bfloat16, 2> {
  uint32_t w;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { w = *reinterpret_cast<const uint32_t*>(p); }
  __device__ __forceinline__ void zero() { w = 0u; }
  __device__ __forceinline__ float operator[](int e) const { return (e & 1) ? bf16_hi(w) : bf16_lo(w); }
};
template <int PER>
struct RowSlice<float, PER> {
  float x[PER];
  __device__ __forceinline__ void load(const float* p) {
    if constexpr (PER == 4) {
      const float4 v = *reinterpret_cast<const float4*>(p);
      x[0] = v.x;
      x[1] = v.y;
      x[2] = v.z;
      x[3] = v.w;
    } else {
      const float2 v = *reinterpret_cast<const float2*>(p);
      x[0] = v.x;
      x[1] = v.y;
    }
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int e = 0; e < PER; ++e) x[e] = 0.f;
  }
  __device__ __forceinline__ float operator[](int e) const { return x[e]; }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---- compress -----------------------------------------------------------------------------
struct SeqTable {
  int32_t n[SELKV_MAX_BATCH];  // prefill length n_b
  int32_t m[SELKV_MAX_BATCH];  // budget m_b = floor(rho * n_b)
  int32_t t1[SELKV_MAX_BATCH];  // tensor-core scoring, pass 1: key tiles of the sequences before b (one KV head)
};

struct ScoreWalk;
struct CompressArgs {
  bool chain;     // launch with launch_chained's early start
  int dtype, B, Hq, Hkv, G, D, W, n_cap, m_cap;
  int R;          // observation rows per KV head: G * W
  int nchunks;    // column chunks of the row-statistics pass
  int row_chunk;  // columns of a chunk (CUDA-core scoring)
  float alpha;
  int pool_kernel, bucket, recent, gate_mode, empty_bucket;
  int per_head;   // SELKV_SELECT_PER_HEAD: selection units are (b, kv), not b
  int rope;       // selkv_rope layout of the kept keys' repositioning (0: off)
  int bias_count; // SELKV_BIAS_COUNT: bias from merge counts instead of ratios
  float rope_theta;
  int rope_hi;    // coarse table entries: position shifts up to 256 * rope_hi
  float2* rope_tab;  // [rope_hi + 256][d/2] (cos, sin) of e * w_f: rows e = 256 c (c < rope_hi), then e = c
  float scale_log2;  // log2(e) / sqrt(d)
  const void* K;
  const void* V;
  const void* Q;
  void* Kc;
  void* Vc;
  float* bias;
  int32_t* lengths;
  // debug outputs (nullable)
  uint8_t* dbg_topk;
  int32_t* dbg_kept_idx;
  int32_t* dbg_target;
  float* dbg_gate;
  uint8_t* dbg_decision;
  float* dbg_ratio;
  // workspace arrays
  uint32_t* flags;
  int32_t* seq_n;
  int32_t* seq_m;
  int32_t* seq_t1;   // [B] SeqTable::t1
  ScoreWalk* p2_walk;  // scoring entry point, tensor cores: pass 2's shares for a call with that pass alone
  float2* rowpart;   // (max, sum) of 2^(s' - max): [B][Hkv][nchunks][R] per column chunk; tensor cores: [pieces][R]
  float2* rowstat;   // [B][Hkv][R] (M, 1 / (G * Z))
  float* attn;       // [B][Hkv][n_cap]
  float* vnorm;      // [B][Hkv][n_cap]
  float* score;      // [B][Hkv][n_cap]
  uint8_t* kflag;    // [units][n_cap] 1 = kept (units: B, or B * Hkv in per-head mode)
  int32_t* slot_of;  // [units][n_cap] slot of a kept position, -1 otherwise
  int32_t* kept_pos; // [units][m_cap] position of each slot
  // Kept masks per 32 positions (bit i: position 32 w + i is kept) and the slot of the first kept
  // one, in the place of kflag and slot_of where merge_uses_mma
  uint2* kmask;      // [units][kmask_ld] (mask, slot)
  int kmask_ld;      // ceil(n_cap / 32)
  int use_kmask;
  int nbk;           // buckets per sequence at n_cap: ceil(n_cap / bucket)
  int32_t* tau;      // [B][Hkv][nbk] merge target of each bucket (-1: no kept token)
  float* atau;       // [B][Hkv][nbk] a of that target
  float* ratio;      // [B][Hkv][m_cap] attention ratio R of each slot
  float* mcount;     // [B][Hkv][m_cap] evicted tokens merged into each slot (g > 0)
  // full cosine routing (routing == SELKV_ROUTE_COSINE)
  int routing;
  int cos_chunks;      // position chunks of the stable counting sort by target slot
  int cos_chunk;       // positions per chunk (a multiple of 32)
  int cos_mpad;        // m_cap rounded up to a whole 256-slot tile
  int32_t* ev_pos;     // [units][n_cap] evicted positions in ascending order
  int32_t* cos_tslot;  // [B][Hkv][n_cap] target slot of an evicted j merged with g > 0, else -1
  float* cos_g;        // [B][Hkv][n_cap] gate g of an evicted j
  float* cos_invn;     // [B][Hkv][cos_mpad] 1 / ||v|| of each slot's kept value (0 for a zero norm)
  int32_t* cos_rank;   // [B][Hkv][n_cap] rank of j among the earlier j of its chunk with its target
  int32_t* cos_order;  // [B][Hkv][n_cap] contributors grouped by target slot, ascending within
  int32_t* cos_cnt;    // [B][Hkv][cos_chunks][m_cap] contributors per (chunk, slot), then their prefix
  int2* cos_seg;       // [B][Hkv][m_cap] (first entry in cos_order, contributors) of each slot
};

// SM count used to plan grids and splits: fixed, so that workspace sizes and results do
// not depend on which device answers (GB300: 152 SMs).
constexpr int kPlanSMs = 152;

// Where each CTA (group) of a tensor-core scoring pass starts in the list of (unit, key tile) pairs,
// and how many tiles it takes.
struct ScoreWalk {
  int32_t u0[kPlanSMs], t0[kPlanSMs], cnt[kPlanSMs];
  int32_t n[kPlanSMs];                      // length of the first unit's sequence
  int32_t part0[kPlanSMs], parts[kPlanSMs];  // pass 2: the first unit's partials of pass 1
  int32_t p1_split, p1_per;  // pass 2: how pass 1 cut the tiles (splits per unit, or 0 and tiles per CTA)
};

// Selection unit of (b, kv): the sequence in the shared mode, the KV head in the per-head mode.
__host__ __device__ __forceinline__ size_t sel_unit(const CompressArgs& a, int b, int kv) {
  return a.per_head ? (size_t)b * a.Hkv + kv : (size_t)b;
}

// Coarse RoPE table entries for caches of n_cap rows: position shifts e < n_cap split as
// e = 256 e_hi + e_lo.
__host__ __device__ constexpr int rope_coarse(int n_cap) { return n_cap / 256 + 1; }

// Columns per CTA in the CUDA-core row-statistics pass: 512 (few partials to fold), halved down to
// a tile of 64 while the CTAs would leave SMs empty (one prompt of 1k with 2 KV heads: 4 CTAs of 512
// columns took 40 us, 32 of 64 take 8).
__host__ __device__ constexpr int score_simt_chunk(int B, int Hkv, int n_cap, int R) {
  int chunk = 512;
  while (chunk > 64 && (long long)B * Hkv * ((R + 63) / 64) * ((n_cap + chunk - 1) / chunk) < kPlanSMs) chunk /= 2;
  return chunk;
}

// Exact radix selection (select_grid.cu).
struct RadixCut {
  uint32_t T;  // bits of the threshold
  int32_t jcut;  // last position taken among the entries equal to T
};
struct SelectWs {
  RadixCut* topk;  // [B * Hkv] each KV head's top-m_s
  uint32_t* tkey;  // [B][n_cap] trim keys, where a span of them does not fit shared memory
};
size_t select_ws_bytes(int B, int Hkv, int n_cap);
SelectWs carve_select_ws(void* base, int B, int Hkv, int n_cap);
cudaError_t launch_select_grid(const CompressArgs& a, const SelectWs& w, cudaStream_t s);

// Scoring: tensor-core path for bf16 with G W <= 256 rows, CUDA-core path otherwise.
bool score_uses_tc(int dtype, int D, int R);
size_t score_tc_partials(int B, int Hkv);  // rows of R partials that pass 1 leaves
int score_tc_tiles1(int n);                // pass-1 key tiles of n keys
// passes: bit 0 = row statistics (pass 1; on CUDA cores also their fold), bit 1 = column sums (pass 2)
constexpr int kScoreRowstats = 1, kScoreColsums = 2, kScoreAll = 3;
cudaError_t launch_score_tc(const CompressArgs& a, const SeqTable& tab, cudaStream_t s, int passes = kScoreAll);
cudaError_t launch_score_simt(const CompressArgs& a, cudaStream_t s, int passes = kScoreAll);
ScoreWalk plan_colsums(const CompressArgs& a, const SeqTable& tab);  // tensor cores: pass 2's shares
cudaError_t launch_seq_setup(const CompressArgs& a, const SeqTable& tab, const ScoreWalk& w, cudaStream_t s);
cudaError_t launch_rowstat_reduce(const CompressArgs& a, cudaStream_t s);
// Routing, merge and kept-row copy in one kernel (merge_mma.cu): bf16, buckets of 32, bucket routing.
bool merge_uses_mma(int dtype, int D, int bucket, int routing);
cudaError_t launch_merge_mma(const CompressArgs& a, cudaStream_t s);
// Compensation averaged across layers (layer_average.cu).
constexpr int kMaxLayers = 128;
struct LayerPtrs {
  const int32_t* kept[kMaxLayers];  // each layer's kept positions [B][units per b][m_cap]
  float* bias[kMaxLayers];          // each layer's bias [B][Hkv][m_cap], read and rewritten
};
struct LayerAvgArgs {
  int B, Hkv, m_cap, n_cap, per_head, L;
  float alpha;
  const int32_t* lengths;  // [B] compressed lengths
  float* acc;              // [B][units per b][n_cap] sum over layers of expm1(bias / alpha)
  uint32_t* flags;
};
cudaError_t launch_layer_average(const LayerAvgArgs& a, const LayerPtrs& P, cudaStream_t s);
// Full cosine routing after the kept rows are in place: argmax, gate, grouping and merge.
cudaError_t launch_route_cosine(const CompressArgs& a, cudaStream_t s);
int cosine_kernels(int dtype, int D);  // kernels launch_route_cosine enqueues
// Chunks of the counting sort for caches of n_cap positions, and the chunk length.
constexpr int kMaxCosChunks = 32;
__host__ __device__ constexpr int cos_chunks_for(int n_cap) {
  return n_cap <= 1024 ? 1 : (n_cap + 1023) / 1024 < kMaxCosChunks ? (n_cap + 1023) / 1024 : kMaxCosChunks;
}
__host__ __device__ constexpr int cos_chunk_len(int n_cap) {
  return ((n_cap + cos_chunks_for(n_cap) - 1) / cos_chunks_for(n_cap) + 31) / 32 * 32;
}

// ---- decode -------------------------------------------------------------------------------
struct DecodeArgs {
  int dtype, B, Hq, Hkv, G, D, m_cap, splits;
  float scale_log2;  // log2(e) / sqrt(d)
  const void* q;
  void* Kc;
  void* Vc;
  float* bias;
  int32_t* lengths;
  const void* k_new;
  const void* v_new;
  void* out;
  uint32_t* flags;
  uint32_t* cnt_head;  // [B][Hkv] arrivals per (b, kv) (self-resetting)
  uint32_t* cnt_seq;   // [B] (b, kv) completions per sequence (self-resetting)
  float* partial;      // [B][Hkv] records of decode_record_floats(G, splits, D) floats
};

// Floats of one (sequence, KV head) record of split partials: the unnormalised outputs
// o [G][S][D], then the (max in base 2, sum) pairs [G][S] padded to a 16-byte multiple, so
// every record starts 16-byte aligned and can be moved with one bulk copy.
__host__ __device__ constexpr size_t decode_record_floats(int G, int S, int D) {
  return (size_t)G * S * D + (((size_t)G * S * 2 + 3) & ~(size_t)3);
}

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per kernel and device (the attribute
// persists; repeating it costs host time on every launch).  Keyed by the kernel itself.
template <auto Kern>
cudaError_t set_smem_once(int bytes) {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit != 0 && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && bit != 0) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

// Once per kernel and device: clusters of more than eight CTAs.
template <auto Kern>
cudaError_t allow_any_cluster_once() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit != 0 && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(Kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && bit != 0) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

// Whether the kernels of a call may be brought up early (launch_chained): on the default stream, where
// nothing else hides their launches.  With several streams, or in a captured graph, the other work
// does (four streams: 0.176 ms a layer either way), and there a decode graph of 8192 nodes replayed
// afterwards took 23.2 us a launch in place of 20.9 in some programs.
inline bool may_chain(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }

// Launch of a kernel that begins with chain_begin (or pdl_wait): it is brought up while its
// predecessor on the stream still runs, which hides its launch (about 1.7 us a kernel: one layer at
// 16k 88 -> 76 us, 1k of fp32 64 -> 45).
template <typename... P, typename... A>
cudaError_t launch_chained(bool chain, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           const A&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// True when the merge kernel copies the kept rows itself (bucket routing, no repositioning),
// so the separate copy kernel is not launched.
bool merge_copies_kept_rows(const CompressArgs& a);

// SELKV_ERR_CUDA, with `e` kept for selkv_last_cuda_error on this thread.
selkv_status cuda_fail(cudaError_t e);

#ifndef SELKV_DEC_UNITS_MAX_ROWS
#define SELKV_DEC_UNITS_MAX_ROWS 2112  // persistent unit-walking decode: most rows of a unit
#endif
// Splits per (b, kv) of a decode launch; unit_walk: the tensor-core decode, which walks many
// short one-split units with persistent CTAs.
int decode_splits(int B, int Hkv, int m_cap, int num_sms, bool unit_walk);
cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t s);     // dispatch by dtype
cudaError_t launch_decode_tc(const DecodeArgs& a, cudaStream_t s);  // bf16: TMA + tensor cores

}  // namespace selkv
