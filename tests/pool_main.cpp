// Test driver of the pool's rule (csrc/pp_pool_host.h): unused, free, total, whether
// the context ends; prints the bytes to keep.
#include <cstdio>
#include <cstdlib>

#include "../paper_2512_12094_gb300/csrc/pp_pool_host.h"

int main(int, char** argv) {
  auto v = [&](int k) { return (size_t)strtoull(argv[k], nullptr, 10); };
  printf("%zu\n", pppool::keep(v(1), v(2), v(3), v(4) != 0));
  return 0;
}
