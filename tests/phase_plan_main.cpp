// Test driver of the phase planner: reads W, the number of gates, max_active,
// max_bits, whether strings are damped, whether triangular runs are wanted, and the occupancy words (x, then z),
// then per gate its activity and its x and z words (decimal); prints the touched
// flags in one line, then "first count kind" (1 commuting, 3 triangular too) and the OR of the generators
// per phase.
#include <cstdio>
#include <vector>

#include "../paper_2512_12094_gb300/csrc/pp_phase.h"

int main() {
  int W, G, bits, damp, tri;
  double active;
  if (scanf("%d %d %lf %d %d %d", &W, &G, &active, &bits, &damp, &tri) != 6) return 1;
  std::vector<uint64_t> occ(2 * W);
  for (int j = 0; j < 2 * W; ++j)
    if (scanf("%llu", (unsigned long long*)&occ[j]) != 1) return 1;
  std::vector<uint64_t> x((size_t)G * W), z((size_t)G * W);
  std::vector<float> act(G);
  for (int g = 0; g < G; ++g) {
    if (scanf("%f", &act[g]) != 1) return 1;
    for (int j = 0; j < W; ++j)
      if (scanf("%llu", (unsigned long long*)&x[g * W + j]) != 1) return 1;
    for (int j = 0; j < W; ++j)
      if (scanf("%llu", (unsigned long long*)&z[g * W + j]) != 1) return 1;
  }
  std::vector<ppphase::Gen> gens(G);
  for (int g = 0; g < G; ++g) gens[g] = {&x[g * W], &z[g * W]};
  const auto touch = ppphase::touched(gens, W, occ.data(), occ.data() + W, damp != 0);
  for (unsigned char t : touch) printf("%d ", t);
  printf("\n");
  ppphase::Limits lim;
  lim.max_active = active;
  lim.max_bits = bits;
  lim.triangular = tri != 0;
  for (const auto& p : ppphase::plan(gens, W, touch.data(), act.data(), lim)) {
    printf("%d %d %d", p.first, p.count, p.commuting + 2 * p.triangular);
    for (int j = 0; j < W; ++j) printf(" %llu", (unsigned long long)p.ux[j]);
    for (int j = 0; j < W; ++j) printf(" %llu", (unsigned long long)p.uz[j]);
    printf("\n");
  }
  return 0;
}
