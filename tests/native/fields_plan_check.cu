// Host-side driver of the workspace plans (csrc/fields_plan.cuh, compiled for the
// CPU).  Reads one plan's arguments per line from stdin and prints its fields.
#include <cstdio>
#include <cstring>
#include "../../paper_1810_07067_gb300/csrc/fields_plan.cuh"

int main() {
  char op[8];
  while (scanf("%7s", op) == 1) {
    if (!strcmp(op, "rhs")) {
      int N, M, n, nrhs;
      if (scanf("%d %d %d %d", &N, &M, &n, &nrhs) != 4) return 1;
      const RhsPlan f = rhs_plan(N, M, n, nrhs, pass_bytes());
      printf("%d %d %d %zu %zu %zu %zu %zu\n", f.ring.nkt, f.ring.nct, f.waves, f.a, f.table, f.cost, f.coef, f.bytes);
    } else if (!strcmp(op, "nf")) {
      long long total;
      int nt, nrhs;
      if (scanf("%lld %d %d", &total, &nt, &nrhs) != 3) return 1;
      const NfPlan f = nf_plan(total, nt, nrhs, pass_bytes());
      printf("%d %d %d %d %d %d %d %d %zu %zu %zu %zu %zu %zu %zu %zu\n", f.na, f.nap, f.np, f.nrt, f.nw, f.nct, f.groups, f.passes, f.a,
             f.r, f.b, f.c, f.y, f.sum, f.sum_group, f.bytes);
    } else if (!strcmp(op, "grid")) {
      int N, M, npol, naz, n, nrhs;
      if (scanf("%d %d %d %d %d %d", &N, &M, &npol, &naz, &n, &nrhs) != 6) return 1;
      const FfoPlan f = ffo_plan(N, M, npol, naz, n, nrhs, pass_bytes());
      printf("%d %d %d %d %d %d %d %d %d %d %d %d %d %zu %zu %zu %zu %zu %zu %zu %zu %zu %zu %zu\n", f.P2, f.ring.nkt,
             f.ring.nct, f.np, f.nrt, f.nps, f.nap, f.nw, f.nct, f.snkt, f.snct, f.swp, f.nkt, f.phase, f.a, f.r, f.b, f.c,
             f.y, f.table, f.cost, f.coef, f.coef_block, f.bytes);
    } else {
      return 1;
    }
  }
  return 0;
}
