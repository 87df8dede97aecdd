// Test driver of the sizing of buckets: reads the strings expected, the factor, fill
// and least buckets of blocks and of warps, and the phases' kinds (1 triangular);
// prints buckets and records per bucket of each.
#include <cstdio>
#include <vector>

#include "../paper_2512_12094_gb300/csrc/pp_phase.h"

int main() {
  double strings, factor;
  ppphase::Workers blocks, warps;
  unsigned long long lb, lw;
  if (scanf("%lf %lf %lf %llu %lf %llu", &strings, &factor, &blocks.fill, &lb, &warps.fill, &lw) != 6) return 1;
  blocks.least = lb;
  warps.least = lw;
  std::vector<ppphase::Phase> phases;
  for (int kind; scanf("%d", &kind) == 1;) {
    phases.emplace_back();
    phases.back().triangular = kind;
  }
  for (const ppphase::Room& r : ppphase::bucket_rooms(phases, strings, blocks, warps, factor))
    printf("%llu %llu\n", (unsigned long long)r.nb, (unsigned long long)r.cg);
  return 0;
}
