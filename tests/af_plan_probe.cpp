// Host test driver of the rule that gives a force system to a cluster or to the
// loop (csrc/af_plan.hpp): reads int32 n, cl, rowptr[n + 1], col from a file and
// prints the choice for FP32 and FP64 and the rule's times.
#include <cstdio>
#include <vector>

#include "af_plan.hpp"

using namespace ibg;

int main(int argc, char** argv) {
  FILE* f = argc == 2 ? std::fopen(argv[1], "rb") : nullptr;
  int32_t h[2];
  if (!f || std::fread(h, 4, 2, f) != 2) return 2;
  const int n = h[0], cl = h[1];
  std::vector<int32_t> rp(n + 1), lo(n, 1), hi(n, 0);
  if (std::fread(rp.data(), 4, rp.size(), f) != rp.size()) return 2;
  std::vector<int32_t> col(rp[n]);
  if (std::fread(col.data(), 4, col.size(), f) != col.size()) return 2;
  for (int r = 0; r < n; ++r)
    if (rp[r] < rp[r + 1]) {
      const auto e = std::minmax_element(col.data() + rp[r], col.data() + rp[r + 1]);
      lo[r] = *e.first, hi[r] = *e.second;
    }
  const AfcRows a{rp.data(), lo.data(), hi.data()};
  std::printf("%d %d", int(afc_takes<float>(a, n, cl)), int(afc_takes<double>(a, n, cl)));
  if (cl > 0) std::printf(" %.0f %.0f %.0f %.0f\n", afc_cluster_ns<float>(a, n, cl), afc_loop_ns<float>(n),
              n <= afc_max_rows<double>(cl) ? afc_cluster_ns<double>(a, n, cl) : 0.0, afc_loop_ns<double>(n));
  return std::fclose(f);
}
