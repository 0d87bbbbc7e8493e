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

// Sequence table alone (the scoring entry point).
__global__ void seq_setup_kernel(SeqTable tab, int32_t* seq_n, int32_t* seq_m, int32_t* seq_t1, int B) {
  pdl_launch_dependents();
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

cudaError_t launch_seq_setup(const CompressArgs& a, const SeqTable& tab, cudaStream_t s) {
  seq_setup_kernel<<<1, 256, 0, s>>>(tab, a.seq_n, a.seq_m, a.seq_t1, a.B);
  return cudaGetLastError();
}

}  // namespace selkv
