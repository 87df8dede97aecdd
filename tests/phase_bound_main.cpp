// Test driver: plans random layers with a bound on the gates of commuting phases
// and on the key bits of the others, and checks every phase against it.  Arguments:
// qubits, gates, support, seed, max_gates, max_plain, max_bits, triangular.  Prints
// the phases of each kind, or a line that says what is wrong.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../paper_2512_12094_gb300/csrc/pp_phase.h"

int main(int argc, char** argv) {
  if (argc != 9) return 1;
  const int n = atoi(argv[1]), G = atoi(argv[2]), support = atoi(argv[3]), W = (n + 63) / 64;
  std::mt19937_64 rng(atoi(argv[4]));
  std::vector<uint64_t> x((size_t)G * W), z((size_t)G * W), occ(W, ~0ull);
  for (int g = 0; g < G; ++g) {
    const int letter = 1 + (int)(rng() % 3);  // runs of one letter commute
    for (int k = 0; k < support; ++k) {
      const int q = (int)(rng() % n), p = rng() % 8 ? letter : 1 + (int)(rng() % 3);
      if (p & 1) x[g * W + q / 64] |= 1ull << (q % 64);
      if (p & 2) z[g * W + q / 64] |= 1ull << (q % 64);
    }
  }
  std::vector<ppphase::Gen> gens(G);
  for (int g = 0; g < G; ++g) gens[g] = {&x[g * W], &z[g * W]};
  const auto touch = ppphase::touched(gens, W, occ.data(), occ.data(), false);
  const std::vector<float> act(G, 0.1f);
  ppphase::Limits lim;
  lim.max_gates = atoi(argv[5]);
  lim.max_plain = atoi(argv[6]);
  lim.max_bits = atoi(argv[7]);
  lim.triangular = atoi(argv[8]) != 0;
  int kinds[3] = {0, 0, 0}, next = 0;
  for (const auto& p : ppphase::plan(gens, W, touch.data(), act.data(), lim)) {
    int bits = 0, gates = 0;
    for (int j = 0; j < W; ++j) bits += __builtin_popcountll(p.ux[j]) + __builtin_popcountll(p.uz[j]);
    for (int g = p.first; g < p.first + p.count; ++g) gates += touch[g];
    if (p.first < next) return printf("gates out of order\n"), 0;
    next = p.first + p.count;
    if (p.triangular && gates > lim.max_gates) return printf("dense phase of %d gates\n", gates), 0;
    if (p.commuting && !p.triangular && gates > lim.max_plain) return printf("phase of %d gates\n", gates), 0;
    if (!p.commuting && gates > 1 && bits > lim.max_bits) return printf("phase of %d bits\n", bits), 0;
    kinds[p.triangular ? 2 : p.commuting ? 1 : 0]++;
  }
  printf("%d %d %d\n", kinds[0], kinds[1], kinds[2]);
  return 0;
}
