// CPU driver for the representatives of Fourier indices (csrc/pf_index.h): for each "L1 L2 L3"
// read from stdin, their number and the list.
#include <cstdio>

#include "pf_index.h"

int main() {
  int L[3];
  while (std::scanf("%d %d %d", L, L + 1, L + 2) == 3) {
    const int n = fock::pf_count(L);
    std::printf("%d", n);
    for (int r = 0; r < n; ++r) std::printf(" %d", fock::pf_index(L, r));
    std::printf("\n");
  }
  return 0;
}
