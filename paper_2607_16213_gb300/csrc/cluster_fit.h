// Largest cluster that can be placed: plain C++, so that the rule can be tested without a device.
#pragma once

namespace selkv {

// `want` (a power of two) halved until places(size) says that a cluster of that many CTAs can run; a
// single CTA needs no placing.
template <typename F>
int fit_cluster(int want, F places) {
  int cs = want;
  while (cs > 1 && !places(cs)) cs /= 2;
  return cs;
}

}  // namespace selkv
