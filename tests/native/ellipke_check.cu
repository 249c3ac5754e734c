// Host-side driver of ellipke (csrc/special.cuh, compiled for the CPU): reads kc per line,
// prints K and E.
#include <cstdio>
#include "../../paper_1810_07067_gb300/csrc/special.cuh"

int main() {
  double kc, K, E;
  while (scanf("%lf", &kc) == 1) {
    ellipke(kc, &K, &E);
    printf("%.17g %.17g\n", K, E);
  }
  return 0;
}
