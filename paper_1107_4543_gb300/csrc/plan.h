// How a lattice's steps are split into launches (host only; shared with the
// host-compiled tests).
#pragma once
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// k_step_rows: strips of at most 30 chunks (32 lanes less two halo chunks; 28
// where V does not divide nx, whose seam lanes borrow idle lanes' slots), of
// equal even width, so that a strip's stores cover whole 32-byte sectors.
inline RowsGeom rows_geom(const Geom &g, int V, int rows) {
  const bool ragged = g.nx % V != 0;
  const int cap = ragged ? 28 : 30;
  RowsGeom r;
  r.strips = (g.nchunks + cap - 1) / cap;
  if (ragged && r.strips == 1 && g.nchunks > 27) r.strips = 2;  // three seam lanes in one strip
  const int w = (g.nchunks + r.strips - 1) / r.strips;
  r.width = std::min(cap, (w + 1) & ~1);
  if (ragged && r.strips == 1) r.width = std::min(r.width, 27);
  r.strips = (g.nchunks + r.width - 1) / r.width;
  r.rows = rows;
  return r;
}

// whether k_step_rows takes the lattice: its seam chunks are assembled from
// whole neighbouring chunks
inline bool rows_fit(const Geom &g, int V) { return g.nx % V == 0 || g.nchunks >= 3; }

// Rows per task: 32 cost 2 (kRowSteps - 1) / 32 of redundant level-1 rows;
// fewer where the tasks would not fill the resident warps (`slots`) a
// quarter more than once (2048^2 FP32: 16 rows 23.2 us per step, 32 rows
// 31.1, 8 rows 24.9).
inline RowsGeom plan_rows(const Geom &g, int V, int slots) {
  const RowsGeom r = rows_geom(g, V, 32);
  const double fit = (double)g.ny * r.strips / (1.25 * slots);
  return rows_geom(g, V, (int)std::max(8.0, std::min(32.0, fit)));
}

// k_step_tile: the split of least estimated time per step with all tiles
// resident at once (one block per SM).  The estimate, in us per launch, is
// 1.2 + 0.05 per tile row loaded + (0.33 + 0.04 per row) for each step, fitted
// to FP32 101^2 (2 .. 8 steps) and 512^2 (2 .. 6 steps) within 10%.
// steps = 0: no split fits.
inline TileGeom plan_tile(const Geom &g, int esize, int sms, double *us_per_step) {
  TileGeom best = {0, 0, 0, 0, 0};
  *us_per_step = 1e30;
  for (int T = 1; T <= kMaxTileSteps; ++T) {
    const int cols = kTileCols - 2 * tile_halo_x(T);
    int ntx = (g.nx + cols - 1) / cols;
    const int bx = ((g.nx + ntx - 1) / ntx + 1) & ~1;
    ntx = (g.nx + bx - 1) / bx;
    if (ntx > sms) continue;
    for (int nty = 1; nty <= std::min(g.ny, sms / ntx); ++nty) {
      const int by = (g.ny + nty - 1) / nty;
      if (nty > 1 && by == (g.ny + nty - 2) / (nty - 1)) continue;  // same split
      if (tile_bytes(by, T, esize) > (size_t)kMaxSmem) continue;
      double us = 1.2 + 0.05 * (by + 2 * T);
      for (int s = 1; s <= T; ++s) us += 0.33 + 0.04 * (by + 2 * (T - s));
      if (us / T < *us_per_step) {
        *us_per_step = us / T;
        best = {bx, by, ntx, (g.ny + by - 1) / by, T};
      }
    }
  }
  return best;
}

// 32- and 16-bit deviation types: tiles where they fit and are estimated
// faster than one launch per step (2.0 + 6.1 us per 2^20 FP32 nodes, 2.7 +
// 4.1 us in 16 bits, measured from 512^2 to 1024^2); else rows for lattices
// whose tasks keep the warps busy (kRowsNodes: below, single steps measured
// as fast); else, and for the FP64 types (bound by FP64 arithmetic, which
// halos only add to), one step per launch.
constexpr double kRowsNodes32 = 1.25e6, kRowsNodes16 = 3.0e6;

inline void plan_lattice(Lattice &L, int sms) {
  L.plan = PLAN_SINGLE;
  if (L.esize == 8) return;
  const double nodes = (double)L.g.nx * L.g.ny;
  double us = 0;
  const TileGeom t = plan_tile(L.g, L.esize, sms, &us);
  const double single = L.esize == 4 ? 2.0 + 5.8e-6 * nodes : 2.7 + 3.9e-6 * nodes;
  if (t.steps > 1 && us < single) {
    L.plan = PLAN_TILE;
    L.tile = t;
  } else if (nodes >= (L.esize == 4 ? kRowsNodes32 : kRowsNodes16) && rows_fit(L.g, L.V)) {
    L.plan = PLAN_ROWS;
    L.rows = plan_rows(L.g, L.V, sms * (L.esize == 4 ? 12 : 8));
  }
}

// Steps of the next launch of n remaining steps: as many as the plan takes,
// without leaving a single step behind k_step_rows (4 = 2 + 2).
inline int next_steps(const Lattice &L, long n) {
  if (L.plan == PLAN_TILE) return (int)std::min<long>(n, L.tile.steps);
  if (L.plan == PLAN_ROWS) return n == 1 ? 1 : (n == 2 || n == 4 ? 2 : kRowSteps);
  return 1;
}

}  // namespace lbm
