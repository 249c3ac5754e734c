// Host-side driver of the far-pair assembly's two-step block (csrc/block.cuh:
// mueller_combine and mueller_block_combined), compiled for the CPU: reads cases
// as block_check.cu does and prints the block through the general combination
// and (where the case is eligible, else the general one again) the specialised.
#include <cstdio>
#include <vector>
#include "../../paper_1810_07067_gb300/csrc/block.cuh"

static cd rd_c() {
  double a = 0, b = 0;
  if (scanf("%lf %lf", &a, &b) != 2) return C(0.0);
  return C(a, b);
}

int main() {
  int ncase = 0;
  if (scanf("%d", &ncase) != 1) return 2;
  for (int q = 0; q < ncase; ++q) {
    int form = 0, M = 0, m = 0;
    double omega = 0, rt, rpt, zpt, rs, rps, zps;
    if (scanf("%d %lf", &form, &omega) != 2) return 2;
    const cd k0 = rd_c(), k1 = rd_c(), eps0 = rd_c(), mu0 = rd_c(), eps1 = rd_c(), mu1 = rd_c();
    if (scanf("%d %d %lf %lf %lf %lf %lf %lf", &M, &m, &rt, &rpt, &zpt, &rs, &rps, &zps) != 8) return 2;
    const int Ms = M + 2;
    std::vector<cd> S(9 * Ms);
    for (auto& v : S) v = rd_c();
    const cd iw = C(0.0, omega);
    AsmParams ap{};
    ap.k0sq = k0 * k0;
    ap.k1sq = k1 * k1;
    if (form == 0) {
      ap.aEJ = C(1.0); ap.aHM = C(-1.0);
      ap.cEM0 = -(iw * eps0); ap.cEM1 = iw * eps1;
      ap.cHJ0 = -(iw * mu0); ap.cHJ1 = iw * mu1;
    } else {
      ap.aEJ = mu0 / eps0; ap.aHM = -(eps0 / mu0);
      ap.cEM0 = -(iw * mu0); ap.cEM1 = iw * mu1;
      ap.cHJ0 = -(iw * eps0); ap.cHJ1 = iw * eps1;
    }
    const bool unit = ap.aEJ.x == 1.0 && ap.aEJ.y == 0.0 && ap.aHM.x == -1.0 && ap.aHM.y == 0.0;
    const bool simple = unit && ap.k0sq.y == 0.0 && ap.k1sq.y == 0.0 && ap.cEM0.x == 0.0 && ap.cEM1.x == 0.0 &&
                        ap.cHJ0.x == 0.0 && ap.cHJ1.x == 0.0;
    printf("%d\n", simple);
    for (int v = 0; v < 2; ++v) {
      std::vector<cd> F(BK_N * Ms);
      for (int mode = 0; mode < Ms; ++mode) {
        cd S9[9];
        for (int f = 0; f < 9; ++f) S9[f] = S[f * Ms + mode];
        if (v == 1 && simple) mueller_combine<true>(S9, ap, 1.0 / rt, rpt, zpt, &F[mode], Ms);
        else mueller_combine<false>(S9, ap, 1.0 / rt, rpt, zpt, &F[mode], Ms);
      }
      cd g[4][4];
      mueller_block_combined(F.data(), Ms, m, ap, v == 1 && unit, 0.5 * rs * rps, 0.5 * rs, rs * zps, 1.0 / rt, rpt,
                             zpt, g);
      for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) printf("%.17g %.17g\n", g[a][b].x, g[a][b].y);
    }
  }
  return 0;
}
