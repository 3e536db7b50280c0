// Host build of the rule that chooses between clusters and the step kernels (csrc/internal.h),
// for the CPU tests: one line of blocks, lattices, fit per query, one answer each.
#include <cstdio>

#include "../../paper_2107_06355_gb300/csrc/internal.h"

int main() {
  int blocks, lattices, fit;
  while (std::scanf("%d %d %d", &blocks, &lattices, &fit) == 3)
    std::printf("%d\n", pplbm::clusters_pay(blocks, lattices, fit) ? 1 : 0);
  return 0;
}
