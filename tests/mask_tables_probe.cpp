// Host test driver: the packed tables of csrc/kuhn_weights.hpp against the weights
// that they hold, over every incident-cell mask.  Prints one line per property:
// name, cases, failures.
#include <cstdio>

#include "kuhn_weights.hpp"

using namespace ibg;

int main() {
  int n = 0, bad = 0;
  for (int m = 0; m < 256; ++m)
    for (int k = 0; k < 15; ++k, ++n) bad += mass_unpack(mass_pack(m), k) != unsigned(mass_weight(m, k));
  std::printf("mass %d %d\n", n, bad);
  n = bad = 0;
  for (int m = 0; m < 256; ++m)
    for (int k = 0; k < 15; ++k)
      for (int e = 0; e < 9; ++e, ++n) bad += trans_unpack(trans_pack(m, k, e / 4), e) != trans_weight(m, k, e / 3, e % 3);
  std::printf("trans %d %d\n", n, bad);
  n = bad = 0;
  int coupled = 0;
  for (int k = 0; k < 15; ++k)
    for (int e = 0; e < 9; ++e, ++n) {
      bool any = false;
      for (int m = 0; m < 256; ++m) any = any || trans_weight(m, k, e / 3, e % 3) != 0;
      bad += any != trans_couples(k, e / 3, e % 3);
      coupled += any;
    }
  std::printf("couples %d %d\n", n, bad);
  std::printf("coupled %d %d\n", coupled, coupled != 99);
  return 0;
}
