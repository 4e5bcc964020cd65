// Host-only driver for split_layers (no GPU needed): reads "ntiles limit c1 c2
// ..." lines on stdin and prints the split plan.
#include <cstdio>

#include "../../paper_2404_04441_gb300/csrc/common.cuh"

int main() {
  char line[4096];
  while (std::fgets(line, sizeof line, stdin)) {
    long long ntiles = 0, limit = 0;
    int off = 0, ch[kMaxLayers], n = 0, c, k;
    if (std::sscanf(line, "%lld %lld%n", &ntiles, &limit, &off) < 2) continue;
    for (const char *p = line + off; n < kPlanLayers && std::sscanf(p, "%d%n", &c, &k) == 1; p += k)
      ch[n++] = c;
    n = split_layers(ch, n, ntiles, limit);
    for (int i = 0; i < n; ++i) std::printf("%d ", ch[i]);
    std::printf("\n");
  }
  return 0;
}
