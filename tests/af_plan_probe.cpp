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
  std::vector<int32_t> rp(n + 1);
  if (std::fread(rp.data(), 4, rp.size(), f) != rp.size()) return 2;
  std::vector<int32_t> col(rp[n]);
  if (std::fread(col.data(), 4, col.size(), f) != col.size()) return 2;
  const int64_t p32 = afc_cluster_ps<float>(rp.data(), col.data(), 0, n, cl);
  const int64_t p64 = afc_cluster_ps<double>(rp.data(), col.data(), 0, n, cl);
  std::printf("%d %d %lld %lld\n", int(afc_takes<float>(n, cl, p32)), int(afc_takes<double>(n, cl, p64)),
              (long long)p32, (long long)p64);
  return std::fclose(f);
}
