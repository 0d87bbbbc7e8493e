// RoPE repositioning of kept keys (Eq. 7) from the tables of rope_table_kernel.
#pragma once

#include "selkv_internal.cuh"

namespace selkv {

// (cos, sin) of e w_f for the N consecutive frequencies f0 .. f0 + N - 1 (f0 and N even),
// from the coarse and the fine row of e.
template <int N>
__device__ __forceinline__ void rope_angles(const CompressArgs& a, int f0, int e, float2 (&cs)[N]) {
  const int half = a.D / 2;
  const float4* h = reinterpret_cast<const float4*>(a.rope_tab + (size_t)(e >> 8) * half + f0);
  const float4* l = reinterpret_cast<const float4*>(a.rope_tab + (size_t)(a.rope_hi + (e & 255)) * half + f0);
#pragma unroll
  for (int t = 0; t < N / 2; ++t) {
    const float4 hv = h[t], lv = l[t];
    cs[2 * t] = make_float2(hv.x * lv.x - hv.y * lv.y, hv.y * lv.x + hv.x * lv.y);
    cs[2 * t + 1] = make_float2(hv.z * lv.z - hv.w * lv.w, hv.w * lv.z + hv.z * lv.w);
  }
}

// Turn the pair (x, y) back by e w_f (from position j to slot j - e).
__device__ __forceinline__ void rope_back(float& x, float& y, float2 cs) {
  const float nx = x * cs.x + y * cs.y, ny = y * cs.x - x * cs.y;
  x = nx;
  y = ny;
}

}  // namespace selkv
