// Prints the cluster kernel's plan for each line of standard input:
//   B R V logit_bytes sm_count smem_per_sm smem_per_block max_cluster ncw C stages
// as "ncw C stages smem ok fits" (host code only, no device needed).
#include <cstdio>

#include "tv_launch.h"

int main() {
  int B, R, V, lb, ncw, C, stages;
  TreeDevice d;
  while (std::scanf("%d %d %d %d %d %d %d %d %d %d %d", &B, &R, &V, &lb, &d.sm_count,
                    &d.smem_per_sm, &d.smem_per_block, &d.max_cluster, &ncw, &C, &stages) == 11) {
    const FusedPlan p = tv_fused_plan(B, R, V, lb, d, ncw, C, stages);
    std::printf("%d %d %d %zu %d %d\n", p.ncw, p.C, p.stages, p.smem, p.ok ? 1 : 0,
                tv_tree_fits(R, V, (size_t)d.smem_per_block) ? 1 : 0);
  }
  return 0;
}
