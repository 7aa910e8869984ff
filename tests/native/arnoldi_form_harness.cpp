// Host harness for the rule that puts the Arnoldi step on one cluster (iter.h: gm_one_cluster): reads lines
// "len gs expire clusters" and prints 0 or 1 each.
#include <cstdint>
#include <cstdio>

#include "iter.h"

int main() {
  long long len;
  int gs, expire, clusters;
  while (std::scanf("%lld %d %d %d", &len, &gs, &expire, &clusters) == 4)
    std::printf("%d\n", lsq::gm_one_cluster(len, gs, expire, clusters) ? 1 : 0);
}
