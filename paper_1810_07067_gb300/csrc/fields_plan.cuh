// Passes and workspace layouts of the products in fields_oz.cu: host arithmetic
// only.  One plan gives the bytes of the block, the places of its parts and the
// most that a pass puts there, for the call that allocates the block and the one
// that fills it alike.
#pragma once
#include <algorithm>
#include <cmath>
#include "ozaki.cuh"

#define FFO_ATILE (OZ_RT * OZ_KT)
#define FFO_ABLOCK (OZ_S * FFO_ATILE)       // bf16 elements per (row tile, k-tile)
#define FFO_NT 32                           // columns of a tile
#define FFO_BTILE (FFO_NT * OZ_KT)
#define FFO_BBLOCK (OZ_S * FFO_BTILE)       // per (column tile, k-tile)
#define FFO_BYTES ((size_t)512 << 20)       // digits of either operand held at a time

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
// FFO_BYTES, at least one.
#define RHS_WAVES 1024
struct RhsPlan {
  RingPlan ring;
  int waves;                    // of a full pass
  size_t a, table, cost, coef;  // offsets of the parts
  size_t bytes;
};
inline RhsPlan rhs_plan(int N, int M, int n_theta, int nrhs) {
  RhsPlan f{};
  f.ring = ring_plan(M, n_theta);
  const size_t most = std::max<size_t>(1, FFO_BYTES / f.ring.a_row_tile * OZ_RT / N);
  f.waves = (int)std::min<size_t>(most, std::min(nrhs, RHS_WAVES));
  const size_t rt = tiles((size_t)f.waves * N, OZ_RT);
  f.table = f.a + up256(rt * f.ring.a_row_tile);
  f.cost = f.table + f.ring.b;
  f.coef = f.cost + f.ring.cost;
  f.bytes = f.coef + up256(rt * f.ring.y_row_tile);
  return f;
}
