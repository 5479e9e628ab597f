// How a lattice's steps are split into launches (host only; shared with the
// host-compiled tests).
#pragma once
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// k_step_rows: segments of about `rows` rows, as even as they go, each a
// sequence of nchunks + 2 halo lane positions, 32 - 2 halo of them to a task
// (the first ones, halo, are no task's own).
inline RowsGeom rows_geom(const Geom &g, int V, int rows) {
  RowsGeom r;
  r.segs = std::max(1, (g.ny + rows / 2) / rows);
  r.rows = (g.ny + r.segs - 1) / r.segs;
  r.segs = (g.ny + r.rows - 1) / r.rows;
  r.halo = g.nx % V != 0 && g.nx % V < kRowSteps ? 2 : 1;
  const int own = 32 - 2 * r.halo;
  const long long pos = (long long)r.segs * (g.nchunks + 2 * r.halo);
  r.tasks = (int)std::min<long long>((pos - 2 * r.halo + own - 1) / own, 1 << 30);
  return r;
}

// whether k_step_rows takes the lattice: its halo chunks are chunks of their
// own, and its positions are 32-bit
inline bool rows_fit(const Geom &g, int V) {
  return (g.nx % V == 0 || g.nchunks >= 3) && (double)g.ny * (g.nchunks + 4) < 4e9;
}

// Rows per segment: 32 cost 2 (kRowSteps - 1) / 32 of redundant level-1 rows;
// fewer where the tasks would not fill the resident warps (`slots`) a
// quarter more than once (2048^2 FP32: 16 rows 23.2 us per step, 32 rows
// 31.1, 8 rows 24.9).
inline RowsGeom plan_rows(const Geom &g, int V, int slots) {
  const double fit = (double)g.ny * (g.nchunks + 2) / 30.0 / (1.25 * slots);
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
// whose tasks keep the warps busy (rows_min_nodes: below, single steps
// measured as fast); else, and for the FP64 types (bound by FP64 arithmetic, which
// halos only add to), one step per launch.
inline double rows_min_nodes(int esize) { return esize == 4 ? 1.25e6 : 3.0e6; }
// resident warps per SM of k_step_rows
inline int rows_warps(int esize) { return esize == 4 ? 12 : 8; }

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
  } else if (nodes >= rows_min_nodes(L.esize) && rows_fit(L.g, L.V)) {
    L.plan = PLAN_ROWS;
    L.rows = plan_rows(L.g, L.V, sms * rows_warps(L.esize));
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
