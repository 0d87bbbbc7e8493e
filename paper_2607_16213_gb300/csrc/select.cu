// Per-call set-up: sequence table, output lengths.
#include "ptx.cuh"
#include "selkv_internal.cuh"

namespace selkv {
namespace {

// Sequence table and output lengths.
__global__ void setup_kernel(SeqTable tab, CompressArgs a) {
  pdl_launch_dependents();
  for (int b = threadIdx.x; b < a.B; b += blockDim.x) {
    a.seq_n[b] = tab.n[b];
    a.seq_m[b] = tab.m[b];
    a.seq_t1[b] = tab.t1[b];
    a.lengths[b] = tab.m[b];
  }
}

// Sequence table and pass 2's shares (the scoring entry point, whose second pass may follow in a call of
// its own).
__global__ void seq_setup_kernel(SeqTable tab, const __grid_constant__ ScoreWalk w, int32_t* seq_n, int32_t* seq_m,
                                 int32_t* seq_t1, ScoreWalk* walk, int B) {
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < (int)(sizeof(ScoreWalk) / 4); i += blockDim.x)
    reinterpret_cast<int32_t*>(walk)[i] = reinterpret_cast<const int32_t*>(&w)[i];
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    seq_n[b] = tab.n[b];
    seq_m[b] = tab.m[b];
    seq_t1[b] = tab.t1[b];
  }
}

}  // namespace

cudaError_t launch_setup(const CompressArgs& a, const SeqTable& tab, cudaStream_t s) {
  setup_kernel<<<1, 256, 0, s>>>(tab, a);
  return cudaGetLastError();
}

cudaError_t launch_seq_setup(const CompressArgs& a, const SeqTable& tab, const ScoreWalk& w, cudaStream_t s) {
  seq_setup_kernel<<<1, 256, 0, s>>>(tab, w, a.seq_n, a.seq_m, a.seq_t1, a.p2_walk, a.B);
  return cudaGetLastError();
}

}  // namespace selkv
