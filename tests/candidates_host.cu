// Host harness for the tuner's candidates (fei_candidates.cuh), driven by
// test_plan_candidates_cpu.py: per line of input "kind ntc sf_too" the pairs
// "variant:grid_cap" on one line.
#include <stdio.h>

#include "fei_candidates.cuh"

int main() {
  int kind, ntc, sf_too;
  while (scanf("%d %d %d", &kind, &ntc, &sf_too) == 3) {
    fei::Candidate c[fei::kMaxCandidates];
    const int n = fei::list_candidates((fei::KernelKind)kind, ntc, sf_too != 0, c);
    for (int i = 0; i < n; ++i) printf("%d:%lld ", c[i].variant, (long long)c[i].grid_cap);
    printf("\n");
  }
  return 0;
}
