// Passes and workspace layouts of the products in fields_oz.cu: host arithmetic
// only.  One plan gives the bytes of the block, the places of its parts and the
// most that a pass puts there, for the call that allocates the block and the one
// that fills it alike.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include "ozaki.cuh"

#define FFO_ATILE (OZ_RT * OZ_KT)
#define FFO_ABLOCK (OZ_S * FFO_ATILE)       // bf16 elements per (row tile, k-tile)
#define FFO_NT 32                           // columns of a tile
#define FFO_BTILE (FFO_NT * OZ_KT)
#define FFO_BBLOCK (OZ_S * FFO_BTILE)       // per (column tile, k-tile)
#define FFO_BYTES ((size_t)512 << 20)       // what a pass holds of an operand's digits, or of sums

// FFO_BYTES; a small bound, so that tests see many passes on small inputs, where the
// environment variable MUELLER_FAULT_INJECT says "small_passes".
inline size_t pass_bytes() {
  const char* v = std::getenv("MUELLER_FAULT_INJECT");
  return v && std::strstr(v, "small_passes") ? (size_t)4 << 20 : FFO_BYTES;
}

inline size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }
inline size_t tiles(size_t v, size_t t) { return (v + t - 1) / t; }

// Ring integrals of rows k N + i, k < count.
struct RingPlan {
  int nkt, nct, E;
  size_t a_row_tile, b, cost, y_row_tile;  // bytes, per 128 rows (a, y) or in all
};
inline RingPlan ring_plan(int M, int n) {
  RingPlan f{};
  f.nkt = (int)tiles(n / 4 + 1, OZ_KT);
  f.nct = (int)tiles(M / 2 + 1 + (M & 1), FFO_NT);  // m = 0, 2, ... (1, 3, ...) up to M + 1
  int e = 0;
  std::frexp(4.0 / n, &e);
  f.E = e + 1;
  f.a_row_tile = (size_t)2 * f.nkt * FFO_ABLOCK * 2;
  f.b = up256((size_t)2 * f.nct * f.nkt * FFO_BBLOCK * 2);
  f.cost = up256((size_t)f.nkt * OZ_KT * 8);
  f.y_row_tile = (size_t)2 * f.nct * FFO_NT * OZ_RT * 8;
  return f;
}

// Ring integrals of plane waves: waves come RHS_WAVES at a time (one table of
// factors) and pass as many of them at once as keep the samples' digits within
// `most` bytes, at least one.
#define RHS_WAVES 1024
struct RhsPlan {
  RingPlan ring;
  int waves;                    // of a full pass
  size_t a, table, cost, coef;  // offsets of the parts
  size_t bytes;
};
inline RhsPlan rhs_plan(int N, int M, int n_theta, int nrhs, size_t most) {
  RhsPlan f{};
  f.ring = ring_plan(M, n_theta);
  const size_t fit = std::max<size_t>(1, most / f.ring.a_row_tile * OZ_RT / N);
  f.waves = (int)std::min<size_t>(fit, std::min(nrhs, RHS_WAVES));
  const size_t rt = tiles((size_t)f.waves * N, OZ_RT);
  f.table = f.a + up256(rt * f.ring.a_row_tile);
  f.cost = f.table + f.ring.b;
  f.coef = f.cost + f.ring.cost;
  f.bytes = f.coef + up256(rt * f.ring.y_row_tile);
  return f;
}

// Far field on a grid.  Passes over the polar angles (np of the upper half: rows (angle,
// cos or sin)) and the sides; the ring integrals of an angle pass come in blocks of nps
// angles, and its products in groups of nap of the M + 2 indices a, where the digits
// of all would not fit `most` bytes (N = 4096, M = 568: 4.8 GB for a row tile of 64 angles).
// The sums over the modes take (side, polar angle) pairs swp at a time.
struct FfoPlan {
  int P2, na, nkt;     // upper angles, indices, k-tiles of nodes
  RingPlan ring;
  int np, nrt, nps, nap;
  int nw, nct;         // sides of a pass and their column tiles
  int snkt, snct, swp;
  size_t phase, a, r, b, c, y, table, cost, coef;  // offsets of the parts
  size_t coef_block;   // bytes of a block's ring integrals
  size_t bytes;
};
inline FfoPlan ffo_plan(int N, int M, int n_polar, int n_azim, int n_alpha, int nrhs, size_t most) {
  FfoPlan f{};
  f.P2 = (n_polar + 1) / 2;
  f.na = M + 2;
  f.nkt = N / OZ_KT;
  f.ring = ring_plan(M, n_alpha);
  const size_t ra = (size_t)f.nkt * FFO_ABLOCK * 2, rb = (size_t)f.nkt * FFO_BBLOCK * 2;  // an index's digits, per tile
  auto fit = [&](size_t each) { return std::max<size_t>(1, most / each); };
  f.nrt = (int)std::min(tiles(2 * (size_t)f.P2, OZ_RT), fit(f.na * ra));
  f.np = (int)std::min<size_t>({(size_t)f.P2, (size_t)f.nrt * OZ_RT / 2, fit(f.ring.y_row_tile * N / OZ_RT)});
  f.nrt = (int)tiles(2 * (size_t)f.np, OZ_RT);
  f.nps = (int)std::min<size_t>(f.np, fit(f.ring.a_row_tile * N / OZ_RT));
  f.nap = (int)std::min<size_t>(f.na, fit(f.nrt * ra));
  const size_t ty = (size_t)f.na * FFO_NT * f.nrt * OZ_RT * 8;  // sums of a column tile
  f.nw = (int)std::max<size_t>(1, std::min<size_t>(nrhs, most / std::max(f.nap * rb, ty) * FFO_NT / 24));
  f.nct = (int)tiles((size_t)24 * f.nw, FFO_NT);
  f.snkt = (int)tiles(M + 1, OZ_KT);
  f.snct = (int)tiles(n_azim / 2 + 1, FFO_NT);
  const size_t sa = (size_t)2 * f.snkt * FFO_ABLOCK * 2, sy = (size_t)2 * f.snct * FFO_NT * OZ_RT * 8;  // per row tile
  f.swp = (int)std::min<size_t>((size_t)nrhs * n_polar, fit(std::max(sa, sy)) * OZ_RT / 6);
  const size_t srt = tiles((size_t)6 * f.swp, OZ_RT), rrt = tiles((size_t)f.nps * N, OZ_RT);
  f.coef_block = rrt * f.ring.y_row_tile;
  f.a = f.phase + up256((size_t)N * ((size_t)f.P2 * 16 + 24));  // and the weights
  f.r = f.a + up256(std::max({(size_t)f.nap * f.nrt * ra, rrt * f.ring.a_row_tile, srt * sa}));
  f.b = f.r + up256(std::max((size_t)f.nap * f.nrt, 2 * srt) * OZ_RT * 8);
  f.c = f.b + up256(std::max((size_t)f.nap * f.nct * rb, (size_t)2 * f.snct * f.snkt * FFO_BBLOCK * 2));
  f.y = f.c + up256((size_t)f.nap * f.nct * FFO_NT * 8);
  f.table = f.y + up256(std::max(f.nct * ty, srt * sy));
  f.cost = f.table + f.ring.b;
  f.coef = f.cost + f.ring.cost;
  f.bytes = f.coef + up256(tiles(f.np, f.nps) * f.coef_block);
  return f;
}

// Fields at points.  The ring points are cut into indices of NF_KC; the rows' digits
// (points), the columns' digits (sides) and the indices' sums are each held for as
// many indices, points and sides at a time as `most` bytes take: all the indices when
// one row tile's digits of all of them fit, else passes over them whose sums add up
// (the sums of all points are kept meanwhile, so that the columns are cut once a pass).
// (A point close to the surface has 8192 azimuths on refined panels, 4e6 ring points:
// 8 GB of digits for one row tile.)
#define NF_KC 512
#define NF_ROWS 18
struct NfPlan {
  int na, nap;             // indices in all, of a ring pass
  int np, nrt;             // points of a pass and their row tiles
  int nw, nct;             // sides of a product and their column tiles
  int groups, passes;      // products of sides and passes of points whose sums are held together
  size_t a, r, b, c, y, sum;  // offsets of the parts
  size_t sum_group;        // values of one product's sums, [pass][group]
  size_t bytes;
};
inline NfPlan nf_plan(long long total, int nt, int nrhs, size_t most) {
  NfPlan f{};
  const size_t ta = (size_t)(NF_KC / OZ_KT) * FFO_ABLOCK * 2, tb = (size_t)(NF_KC / OZ_KT) * FFO_BBLOCK * 2;
  const size_t ty = (size_t)FFO_NT * OZ_RT * 8;  // an index's digits of a row tile, a column tile, its sums of both
  const size_t fit = std::max<size_t>(1, most / ta);  // (index, row tile) pairs held
  f.na = (int)tiles((size_t)total, NF_KC);
  const size_t all = tiles((size_t)NF_ROWS * nt, OZ_RT);
  f.nrt = (int)std::min(all, (size_t)f.na <= fit ? fit / f.na : (size_t)4);
  f.np = std::min(nt, f.nrt * OZ_RT / NF_ROWS);
  f.np = (int)tiles(nt, tiles(nt, f.np));  // equal passes
  f.nrt = (int)tiles((size_t)NF_ROWS * f.np, OZ_RT);
  f.nap = (int)tiles(f.na, tiles(f.na, std::max<size_t>(1, fit / f.nrt)));
  const size_t ct = std::min(most / (f.nap * tb), most / (f.nap * (size_t)f.nrt * ty));
  f.nw = (int)std::min<size_t>(nrhs, std::max<size_t>(1, ct * FFO_NT / 12));
  f.nct = (int)tiles((size_t)12 * f.nw, FFO_NT);
  f.sum_group = (size_t)f.nct * FFO_NT * f.nrt * OZ_RT;
  f.groups = (int)std::min(tiles(nrhs, f.nw), std::max<size_t>(1, most / (f.sum_group * 8)));
  f.passes = (int)std::min(tiles(nt, f.np), std::max<size_t>(1, most / (f.groups * f.sum_group * 8)));
  f.r = f.a + up256((size_t)f.nap * f.nrt * ta);
  f.b = f.r + up256((size_t)f.nap * f.nrt * OZ_RT * 8);
  f.c = f.b + up256((size_t)f.nap * f.nct * tb);
  f.y = f.c + up256((size_t)f.nap * f.nct * FFO_NT * 8);
  f.sum = f.y + up256((size_t)f.nap * f.sum_group * 8);
  f.bytes = f.sum + up256(f.passes * f.groups * f.sum_group * 8);
  return f;
}
