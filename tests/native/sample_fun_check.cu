// Host-side driver of the sample functions (csrc/special.cuh), compiled for the
// CPU: reads "xre xim" per line and prints c, sinc, sig1, sig2, a, eta of the
// complex form, then of the real form at xre ("re im" each).
#include <cstdio>
#include "../../paper_1810_07067_gb300/csrc/special.cuh"

int main() {
  SeriesTables T;
  fill_series_tables(&T);
  double a, b;
  while (scanf("%lf %lf", &a, &b) == 2) {
    const cd x = C(a, b), xi = C(1.0) / x;
    cd s, c;
    csincos(x, &s, &c);
    const SampleFun<cd> f = cabs(x) < 2.0 ? sample_series<cd>(T, x * x) : sample_closed<cd>(s, c, xi, xi * xi);
    const SampleFun<double> r = std::fabs(a) < 2.0 ? sample_series<double>(T, a * a)
                                                   : sample_closed<double>(std::sin(a), std::cos(a), 1 / a, 1 / (a * a));
    const cd v[6] = {f.c, f.sinc, f.sig1, f.sig2, f.a, f.eta};
    const double w[6] = {r.c, r.sinc, r.sig1, r.sig2, r.a, r.eta};
    for (int q = 0; q < 6; ++q) printf("%.17g %.17g ", v[q].x, v[q].y);
    for (int q = 0; q < 6; ++q) printf("%.17g 0 ", w[q]);
    printf("\n");
  }
  return 0;
}
