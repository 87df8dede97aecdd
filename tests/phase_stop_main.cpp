// Test driver: plans the gates of an all-to-all layer (XX, YY, ZZ on every pair of n
// sites) with and without a limit on the number of phases.  Prints the phases of the
// whole plan and of the limited one, and whether the latter is the former's beginning.
#include <cstdio>
#include <cstdlib>

#include "../paper_2512_12094_gb300/csrc/pp_phase.h"

int main(int argc, char** argv) {
  if (argc != 3) return 1;
  const int n = atoi(argv[1]);
  std::vector<uint64_t> x, z;
  for (int a = 0; a < n; ++a)
    for (int b = a + 1; b < n; ++b)
      for (int p = 0; p < 3; ++p) {
        const uint64_t m = (1ull << a) | (1ull << b);
        x.push_back(p < 2 ? m : 0);
        z.push_back(p > 0 ? m : 0);
      }
  std::vector<ppphase::Gen> gens;
  for (size_t g = 0; g < x.size(); ++g) gens.push_back({&x[g], &z[g]});
  const std::vector<unsigned char> touch(x.size(), 1);
  const std::vector<float> act(x.size(), 0.3f);
  ppphase::Limits lim;
  const auto whole = ppphase::plan(gens, 1, touch.data(), act.data(), lim);
  lim.max_phases = (size_t)atoi(argv[2]);
  const auto part = ppphase::plan(gens, 1, touch.data(), act.data(), lim);
  bool same = part.size() <= whole.size();
  for (size_t k = 0; same && k < part.size(); ++k)
    same = part[k].first == whole[k].first && part[k].count == whole[k].count;
  printf("%zu %zu %d\n", whole.size(), part.size(), (int)same);
  return 0;
}
