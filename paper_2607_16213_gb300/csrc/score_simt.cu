// Observation-window scoring on CUDA cores (fp32 arithmetic for both storage dtypes).
//
// Per (sequence b, KV head kv) the G query heads' W window rows are stacked into R = G * W
// rows.  Row r = g * W + i is query head kv * G + g at position p = n_b - W + i and sees the
// keys j <= p (the causal re-pass of Sec. 3.1).  The cumulative attention of Eq. 5,
// averaged over the group,
//     a_j = (1/G) sum_r 2^(s'_rj - M_r) / Z_r,     s'_rj = log2(e) q_r . k_j / sqrt(d),
// needs each row's normaliser before any column can be summed, so the scores are computed
// twice: pass 1 gathers per-row (max, sum) over column chunks, a small kernel folds the
// chunks, and pass 2 recomputes the same tiles and sums columns.  Both passes use the same
// tile code, so pass 2 sees bit-identical scores.
#include <algorithm>

#include "ptx.cuh"
#include "selkv_internal.cuh"

namespace selkv {

cudaError_t launch_rowstat_reduce(const CompressArgs& a, cudaStream_t s);

namespace {

constexpr int kTile = 64;   // rows and columns per tile
constexpr int kDc = 32;     // head-dimension slice staged in shared memory

// acc[i][j] = q_{r0 + 4ty + i} . k_{c0 + 4tx + j} for a 64 x 64 tile.
template <typename T, int D>
__device__ __forceinline__ void score_tile(const CompressArgs& a, int b, int kv, int n, int r0,
                                           int c0, float (&Qs)[kDc][kTile + 4],
                                           float (&Ks)[kDc][kTile + 4], float (&acc)[4][4]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const int lrow = tid >> 2, ldd = (tid & 3) * 8;
  for (int dc = 0; dc < D; dc += kDc) {
    float x[8];
    const int r = r0 + lrow;
    if (r < a.R) {
      const int h = kv * a.G + r / a.W, i = r % a.W;
      load8(static_cast<const T*>(a.Q) + (((size_t)b * a.Hq + h) * a.W + i) * D + dc + ldd, x);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) Qs[ldd + k][lrow] = x[k];
    const int col = c0 + lrow;
    if (col < n) {
      load8(static_cast<const T*>(a.K) + (((size_t)b * a.Hkv + kv) * a.n_cap + col) * D + dc + ldd, x);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) Ks[ldd + k][lrow] = x[k];
    __syncthreads();
#pragma unroll 8
    for (int dd = 0; dd < kDc; ++dd) {
      const float4 q4 = *reinterpret_cast<const float4*>(&Qs[dd][ty * 4]);
      const float4 k4 = *reinterpret_cast<const float4*>(&Ks[dd][tx * 4]);
      const float qv[4] = {q4.x, q4.y, q4.z, q4.w};
      const float kvv[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(qv[i], kvv[j], acc[i][j]);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ float reduce16_max(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float reduce16_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Pass 1: grid (column chunk, row tile, b * Hkv); per row the (max, sum) of 2^(s' - max)
// over the chunk's visible columns.
template <typename T, int D>
__global__ __launch_bounds__(256) void rowstats_kernel(CompressArgs a) {
  chain_begin();
  __shared__ __align__(16) float Qs[kDc][kTile + 4];
  __shared__ __align__(16) float Ks[kDc][kTile + 4];
  const int chunk = blockIdx.x, r0 = blockIdx.y * kTile, bk = blockIdx.z;
  const int b = bk / a.Hkv, kv = bk % a.Hkv;
  const int n = a.seq_n[b];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float m_run[4], l_run[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { m_run[i] = -INFINITY; l_run[i] = 0.f; }
  const int c_begin = chunk * a.row_chunk;
  const int c_end = min(n, c_begin + a.row_chunk);
  for (int c0 = c_begin; c0 < c_end; c0 += kTile) {
    float acc[4][4];
    score_tile<T, D>(a, b, kv, n, r0, c0, Qs, Ks, acc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + ty * 4 + i;
      const int p = n - a.W + (r % a.W);
      float sv[4], tmax = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = c0 + tx * 4 + j;
        const bool ok = r < a.R && col < n && col <= p;
        sv[j] = ok ? acc[i][j] * a.scale_log2 : -INFINITY;
        tmax = fmaxf(tmax, sv[j]);
      }
      tmax = reduce16_max(tmax);
      const float m_new = fmaxf(m_run[i], tmax);
      float ssum = 0.f;
      if (m_new != -INFINITY) {
#pragma unroll
        for (int j = 0; j < 4; ++j) ssum += exp2f(sv[j] - m_new);
      }
      ssum = reduce16_sum(ssum);
      if (m_new != -INFINITY) {
        l_run[i] = l_run[i] * exp2f(m_run[i] - m_new) + ssum;
        m_run[i] = m_new;
      }
    }
  }
  if (tx == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + ty * 4 + i;
      if (r < a.R) a.rowpart[((size_t)bk * a.nchunks + chunk) * a.R + r] = make_float2(m_run[i], l_run[i]);
    }
  }
}

// Fold of the column chunks of row idx: (M, 1 / (G * Z)).
__device__ __forceinline__ void fold_row(const CompressArgs& a, int idx) {
  if (idx >= a.B * a.Hkv * a.R) return;
  const int r = idx % a.R, bk = idx / a.R;
  const int nch = a.nchunks;  // chunks without visible columns hold (-inf, 0)
  const float2* part = a.rowpart + (size_t)bk * a.nchunks * a.R + r;
  float M = -INFINITY;
#pragma unroll 8
  for (int c = 0; c < nch; ++c) M = fmaxf(M, part[(size_t)c * a.R].x);
  float Z = 0.f;
#pragma unroll 8
  for (int c = 0; c < nch; ++c) {
    const float2 p = part[(size_t)c * a.R];
    if (p.x != -INFINITY) Z += p.y * exp2f(p.x - M);
  }
  a.rowstat[idx] = make_float2(M, 1.f / ((float)a.G * Z));
}

__global__ void rowstat_reduce_kernel(CompressArgs a) {
  chain_begin();
  fold_row(a, blockIdx.x * blockDim.x + threadIdx.x);
}

// The fold in the first `fold_blocks` CTAs and ||v_j|| of Eq. 1 in the others: two kernels' work
// that does not depend on one another in one launch.  D / 8 lanes per row (at most 16), each
// loading 8 elements at a time.
template <typename T, int D>
__global__ __launch_bounds__(256) void fold_norm_kernel(CompressArgs a, int fold_blocks) {
  chain_begin();
  if ((int)blockIdx.x < fold_blocks) {
    fold_row(a, blockIdx.x * blockDim.x + threadIdx.x);
    return;
  }
  constexpr int EPL = 8;                            // elements per load8
  constexpr int LPR = D / EPL < 16 ? D / EPL : 16;  // lanes per row
  constexpr int RPW = 32 / LPR;                     // rows per warp step
  const int lane = threadIdx.x & 31, sub = lane / LPR, sl = lane % LPR;
  const size_t total = (size_t)a.B * a.Hkv * a.n_cap;
  const size_t nwarps = (size_t)(gridDim.x - fold_blocks) * (blockDim.x / 32);
  const size_t warp = ((blockIdx.x - fold_blocks) * (size_t)blockDim.x + threadIdx.x) / 32;
  for (size_t row0 = warp * RPW; row0 < total; row0 += nwarps * RPW) {
    const size_t row = row0 + sub;
    float s = 0.f;
    bool ok = false;
    if (row < total) {
      const int j = (int)(row % a.n_cap);
      const int b = (int)(row / a.n_cap) / a.Hkv;
      ok = j < a.seq_n[b];
      if (ok) {
        const T* p = static_cast<const T*>(a.V) + row * D;
#pragma unroll
        for (int d = sl * EPL; d < D; d += LPR * EPL) {
          float x[8];
          load8(p + d, x);
#pragma unroll
          for (int e = 0; e < 8; ++e) s = fmaf(x[e], x[e], s);
        }
      }
    }
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (ok && sl == 0) a.vnorm[row] = sqrtf(s);
  }
}

// Pass 2: grid (column tile, b * Hkv); a_j = sum_r 2^(s'_rj - M_r) / (G Z_r).
template <typename T, int D>
__global__ __launch_bounds__(256) void colsum_kernel(CompressArgs a) {
  chain_begin();
  __shared__ __align__(16) float Qs[kDc][kTile + 4];
  __shared__ __align__(16) float Ks[kDc][kTile + 4];
  __shared__ float red[16][kTile];
  const int c0 = blockIdx.x * kTile, bk = blockIdx.y;
  const int b = bk / a.Hkv, kv = bk % a.Hkv;
  const int n = a.seq_n[b];
  if (c0 >= n) return;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float colacc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int r0 = 0; r0 < a.R; r0 += kTile) {
    float acc[4][4];
    score_tile<T, D>(a, b, kv, n, r0, c0, Qs, Ks, acc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + ty * 4 + i;
      if (r >= a.R) continue;
      const float2 st = a.rowstat[(size_t)bk * a.R + r];
      const int p = n - a.W + (r % a.W);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = c0 + tx * 4 + j;
        if (col < n && col <= p) colacc[j] += exp2f(acc[i][j] * a.scale_log2 - st.x) * st.y;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) red[ty][tx * 4 + j] = colacc[j];
  __syncthreads();
  if (threadIdx.x < kTile) {
    float s = 0.f;
#pragma unroll
    for (int t = 0; t < 16; ++t) s += red[t][threadIdx.x];
    const int col = c0 + threadIdx.x;
    if (col < n) a.attn[(size_t)bk * a.n_cap + col] = s;
  }
}

template <typename T, int D>
cudaError_t launch_score_t(const CompressArgs& a, cudaStream_t s, int passes) {
  const int row_tiles = (a.R + kTile - 1) / kTile;
  if (passes & kScoreRowstats) {
    launch_chained(a.chain, rowstats_kernel<T, D>, dim3(a.nchunks, row_tiles, a.B * a.Hkv), 256, 0, s, a);
    if (a.V == nullptr) {
      launch_rowstat_reduce(a, s);
    } else {
      const size_t rows = (size_t)a.B * a.Hkv * a.n_cap;
      const int fold = (a.B * a.Hkv * a.R + 255) / 256, norm = (int)std::min<size_t>((rows + 15) / 16, 152 * 8);
      launch_chained(a.chain, fold_norm_kernel<T, D>, fold + norm, 256, 0, s, a, fold);
    }
  }
  if (passes & kScoreColsums)
    launch_chained(a.chain, colsum_kernel<T, D>, dim3((a.n_cap + kTile - 1) / kTile, a.B * a.Hkv), 256, 0, s, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rowstat_reduce(const CompressArgs& a, cudaStream_t s) {
  const int nrows = a.B * a.Hkv * a.R;
  launch_chained(a.chain, rowstat_reduce_kernel, (nrows + 255) / 256, 256, 0, s, a);
  return cudaGetLastError();
}

cudaError_t launch_score_simt(const CompressArgs& a, cudaStream_t s, int passes) {
  if (a.dtype == SELKV_BF16)
    return a.D == 128 ? launch_score_t<__nv_bfloat16, 128>(a, s, passes) : launch_score_t<__nv_bfloat16, 64>(a, s, passes);
  return a.D == 128 ? launch_score_t<float, 128>(a, s, passes) : launch_score_t<float, 64>(a, s, passes);
}

}  // namespace selkv
