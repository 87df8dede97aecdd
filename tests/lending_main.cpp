// Test driver of the server's rule for memory lent to a layer (csrc/pp_admission.h):
// reads budget, reserved, extra, growing, running, slots and the queued jobs'
// reservations from the command line; prints 1 or 0.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_2512_12094_gb300/csrc/pp_admission.h"

int main(int argc, char** argv) {
  auto v = [&](int k) { return strtoull(argv[k], nullptr, 10); };
  std::vector<size_t> queued;
  for (int k = 7; k < argc; ++k) queued.push_back(v(k));
  printf("%d\n", (int)ppadm::may_lend(v(1), v(2), v(3), (int64_t)v(4), (int64_t)v(5), (int)v(6), queued));
  return 0;
}
