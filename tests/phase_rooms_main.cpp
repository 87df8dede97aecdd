// Test driver of the sizing of buckets: reads the terms of the table, the last
// growth, the strings possible, the factor, fill and least buckets of blocks and of
// warps, and the phases' kinds (1 triangular); prints the strings expected and, for
// each phase, its buckets and records per bucket.
#include <cstdio>
#include <vector>

#include "../paper_2512_12094_gb300/csrc/pp_phase.h"

int main() {
  double growth, possible, factor;
  unsigned long long terms;
  ppphase::Workers blocks, warps;
  unsigned long long lb, lw;
  if (scanf("%llu %lf %lf %lf %lf %llu %lf %llu", &terms, &growth, &possible, &factor, &blocks.fill, &lb,
            &warps.fill, &lw) != 8)
    return 1;
  blocks.least = lb;
  warps.least = lw;
  std::vector<ppphase::Phase> phases;
  for (int kind; scanf("%d", &kind) == 1;) {
    phases.emplace_back();
    phases.back().triangular = kind;
  }
  const ppphase::Expected e = ppphase::expected(terms, growth, possible);
  printf("%.17g %.17g\n", e.strings, e.lumps);
  for (const ppphase::Room& r : ppphase::bucket_rooms(phases, e, blocks, warps, factor))
    printf("%llu %llu\n", (unsigned long long)r.nb, (unsigned long long)r.cg);
  return 0;
}
