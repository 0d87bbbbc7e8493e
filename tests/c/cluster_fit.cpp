// The rule for the cluster size, with made-up devices.
#include <cstdio>

#include "cluster_fit.h"

#define CHECK(x)                                  \
  do {                                            \
    if (!(x)) {                                   \
      std::printf("line %d: %s\n", __LINE__, #x); \
      return 1;                                   \
    }                                             \
  } while (0)

int main() {
  for (int most = 0; most <= 32; ++most)      // a device that places up to `most` CTAs together
    for (int want = 1; want <= 16; want *= 2) {
      const int cs = selkv::fit_cluster(want, [&](int size) { return size <= most; });
      CHECK(cs >= 1 && cs <= want);
      CHECK(cs == 1 || cs <= most);
      CHECK(cs == want || 2 * cs > most);      // no larger one of them fits
    }
  std::printf("done\n");
  return 0;
}
