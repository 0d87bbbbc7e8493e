// Per-call set-up: sequence table, output lengths, the selection's initial states.
#include "selkv_internal.cuh"

namespace selkv {
namespace {

// Sequence table, output lengths and the selection's initial radix states.
__global__ void setup_kernel(SeqTable tab, CompressArgs a, SelectWs w) {
  for (int b = threadIdx.x; b < a.B; b += blockDim.x) {
    a.seq_n[b] = tab.n[b];
    a.seq_m[b] = tab.m[b];
    a.lengths[b] = tab.m[b];
  }
  const int units = a.B * a.Hkv;
  for (int i = threadIdx.x; i < units + a.B; i += blockDim.x) {
    const int b = i >= units ? i - units : i / a.Hkv;
    select_init_state(a, w, i, tab.n[b], tab.m[b]);
  }
}

// Sequence table alone (the scoring entry point).
__global__ void seq_setup_kernel(SeqTable tab, int32_t* seq_n, int32_t* seq_m, int B) {
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    seq_n[b] = tab.n[b];
    seq_m[b] = tab.m[b];
  }
}

}  // namespace

cudaError_t launch_setup(const CompressArgs& a, const SeqTable& tab, const SelectWs& w, cudaStream_t s) {
  setup_kernel<<<1, 256, 0, s>>>(tab, a, w);
  return cudaGetLastError();
}

cudaError_t launch_seq_setup(const CompressArgs& a, const SeqTable& tab, cudaStream_t s) {
  seq_setup_kernel<<<1, 256, 0, s>>>(tab, a.seq_n, a.seq_m, a.B);
  return cudaGetLastError();
}

}  // namespace selkv
