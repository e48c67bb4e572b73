// Host driver of the digit engine's selection rule (csrc/oz_rule.h).
// stdin: lines "M N batches groups K_0 .. K_{groups-1}"; stdout: 1 or 0 per line.
#include <cstdio>
#include <vector>

#include "../paper_1905_01331_gb300/csrc/oz_rule.h"

int main() {
  int M, N, groups;
  long long batches;
  while (std::scanf("%d %d %lld %d", &M, &N, &batches, &groups) == 4) {
    std::vector<int> K(groups);
    for (int& k : K) std::scanf("%d", &k);
    std::printf("%d\n", ttn::oz_worth(M, N, batches, K.data(), groups) ? 1 : 0);
  }
  return 0;
}
