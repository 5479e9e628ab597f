// How a lattice's steps are split into launches (host only; shared with the
// host-compiled tests).
#pragma once
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// k_step_rows: segments of about `rows` rows, as even as they go, each a
// sequence of nchunks + 2 halo lane positions, 32 - 2 halo of them to a task
// (the first ones, halo, are no task's own).
inline RowsGeom rows_geom(const Geom &g, int rows) {
  constexpr int V = kRowsV;
  RowsGeom r;
  r.segs = std::max(1, (g.ny + rows / 2) / rows);
  r.rows = (g.ny + r.segs - 1) / r.segs;
  r.segs = (g.ny + r.rows - 1) / r.rows;
  r.halo = g.nx % V != 0 && g.nx % V < kRowSteps ? 2 : 1;
  const int own = 32 - 2 * r.halo;
  const long long pos = (long long)r.segs * (rows_chunks(g) + 2 * r.halo);
  r.tasks = (int)std::min<long long>((pos - 2 * r.halo + own - 1) / own, 1 << 30);
  return r;
}

// whether k_step_rows takes the lattice: its halo chunks are chunks of their
// own, and its positions are 32-bit
inline bool rows_fit(const Geom &g) {
  return (g.nx % kRowsV == 0 || rows_chunks(g) >= 3) && (double)g.ny * (rows_chunks(g) + 4) < 4e9;
}

// resident warps per SM of k_step_rows; k_rows_batch's FP32 form holds 12 (136
// registers), which its fitted rate contains
constexpr int kRowsWarps = 16;

// Work of k_step_rows over a lattice, or summed over a batch's: its tasks and
// the nodes they compute per step (idle lanes, halo lanes and rows included).
struct RowsWork {
  double tasks = 0, nodes = 0;
  void add(const RowsGeom &r) {
    tasks += r.tasks;
    nodes += (double)r.tasks * 32 * kRowsV * (r.rows + kRowSteps - 1);
  }
};

// Estimated us per step: 285 (FP32) or 300 (16 bits) such nodes per ns with
// all warp slots busy, less where there are few tasks per slot.  Measured /
// estimated: 8192^2 276 / 277 FP32 and 262 / 262 FP16, 1024^2 FP32 7.3 / 7.7,
// 700^2 FP32 4.7 / 5.1, 4097 x 3071 FP16 59.6 / 59, 2500 x 2001 FP16 26 /
// 24.6.
inline double rows_us(const RowsWork &w, int esize, int sms, double half = 0.25) {
  const double per_slot = w.tasks / ((double)sms * kRowsWarps);
  const double rate = (esize == 4 ? 285e3 : 300e3) * per_slot / (per_slot + half);
  return w.nodes / rate;
}

// The same for a batch (k_rows_batch): its constants come from shared memory,
// and where it has more than a task or two per slot, short segments fill the
// tail.
// The factors were fitted on one batch (rows_batch_margin has others): measured
// / estimated, 128 lattices of 32^2 .. 1024^2: FP32 in segments of 8, 16, 28, 32
// rows 91 / 83, 85 / 79, 81 / 77, 81 / 77 us, FP16 83 / 79, 80 / 74, 78 / 73,
// 79 / 73.
inline double rows_batch_us(const RowsWork &w, int esize, int sms) {
  return std::max(rows_us(w, esize, sms), 1.15 * rows_us(w, esize, sms, 0.1));
}

// What rows must be estimated to save of a batch's single steps.  5%, but 8%
// in FP16 with fewer than 1.5 tasks per slot: the estimate does not see the
// tail of the second wave there, and FP16's single steps are the fastest ones.
// Measured rows / single steps at estimates of 0.93 and 0.92: 12 lattices of
// 300^2 .. 1000^2 (1.0 tasks per slot) 30.4 / 29.0, 64 of 82^2 .. 1024^2 (1.25)
// 57.0 / 56.4 us; at 0.91, 2000^2 (0.86) 23.3 / 24.5, 0.93, 400 of 85^2 ..
// 300^2 (1.8) 86.9 / 93.8.
inline double rows_batch_margin(const RowsWork &w, bool f16, int sms) {
  return f16 && w.tasks < 1.5 * sms * kRowsWarps ? 0.92 : 0.95;
}

// Estimated us of one single-step launch over `nodes` nodes: its latency and
// the L2's rate while both buffers fit there, HBM's beyond.  Measured: FP32
// 1024^2 8.4, 1500 x 1111 16.4, 2048^2 45; 16 bits 1500 x 1111 9.4, 1732^2
// 17.5, 2048^2 24.5 us.
inline double single_us(double nodes, int esize) {
  const double m = nodes * 1e-6;
  return esize == 4 ? std::max(2.0 + 6.0 * m, 10.8 * m - 2.0) : std::max(2.7 + 3.9 * m, 5.7 * m);
}

// The segment heights tried: low ones cost redundant rows (2 (kRowSteps - 1)
// per segment), high ones leave too few tasks.
constexpr int kRowChoices[] = {8, 12, 16, 24, 32};
constexpr int kBatchRowChoices[] = {8, 12, 16, 20, 24, 28, 32};

// k_step_rows' best split of one lattice and its estimate (rows = 0: the
// lattice does not fit it)
inline RowsGeom plan_rows(const Geom &g, int esize, int sms, double *us) {
  RowsGeom best = {};
  *us = 1e30;
  if (!rows_fit(g)) return best;
  for (int rows : kRowChoices) {
    const RowsGeom r = rows_geom(g, rows);
    RowsWork w;
    w.add(r);
    const double t = rows_us(w, esize, sms);
    if (t < *us) {
      *us = t;
      best = r;
    }
  }
  return best;
}

// Estimated us of one k_step_tile launch of T steps on tiles of `by` rows: 1.2
// + 0.05 per tile row loaded + (0.33 + 0.04 per row) for each step, fitted to
// FP32 101^2 (2 .. 8 steps) and 512^2 (2 .. 6 steps) within 10%.
inline double tile_us(int by, int T) {
  double us = 1.2 + 0.05 * (by + 2 * T);
  for (int s = 1; s <= T; ++s) us += 0.33 + 0.04 * (by + 2 * (T - s));
  return us;
}

// k_step_tile: the split of least estimated time per step with all tiles
// resident at once (one block per SM); steps = 0: no split fits.
inline TileGeom plan_tile(const Geom &g, int esize, int sms, double *us_per_step) {
  TileGeom best = {0, 0, 0, 0, 0};
  *us_per_step = 1e30;
  for (int T = 1; T <= kMaxTileSteps; ++T) {
    const int cols = kTileCols - 2 * tile_halo_x(T);
    int ntx = (g.nx + cols - 1) / cols;
    const int bx = ((g.nx + ntx - 1) / ntx + 1) & ~1;
    ntx = (g.nx + bx - 1) / bx;
    if (ntx > sms) continue;
    // both the estimate and the tile's size grow with its height: the lowest
    // tiles that are resident at once
    const int nty = std::min(g.ny, sms / ntx);
    const int by = (g.ny + nty - 1) / nty;
    if (tile_bytes(by, T, esize) > (size_t)kMaxSmem) continue;
    const double us = tile_us(by, T);
    if (us / T < *us_per_step) {
      *us_per_step = us / T;
      best = {bx, by, ntx, (g.ny + by - 1) / by, T};
    }
  }
  return best;
}

// The least steps that k_step_tile takes: a launch of few steps still pays for
// loading the halo of tall tiles.  Single steps outside a graph cost a little
// more than estimated, so they have to be estimated 25% faster.  us per call of
// 1, 2, 3 steps, tiles / single steps: 700^2 FP16 7.3 / 4.5, 9.9 / 9.0, 12.7 /
// 13.5; one step of 5 x 3000 FP32 4.4 / 2.6, of 512^2 FP32 5.5 / 3.5.
inline int tile_least(const TileGeom &t, double single) {
  int n = 1;
  while (n < t.steps && tile_us(t.by, n) > 1.25 * n * single) ++n;
  return n;
}

// The estimated fastest of tiles, rows and single steps for the 32- and
// 16-bit deviation types (several steps per launch only where they save at
// least 5%); one step per launch for the FP64 types, which FP64 arithmetic
// bounds and halos would only add to.
inline void plan_lattice(Lattice &L, int sms) {
  L.plan = PLAN_SINGLE;
  if (L.esize == 8) return;
  const double single = single_us((double)L.g.nx * L.g.ny, L.esize);
  double best = 0.95 * single, us = 0;
  const TileGeom t = plan_tile(L.g, L.esize, sms, &us);
  if (t.steps > 1 && us < best) {
    L.plan = PLAN_TILE;
    L.tile = t;
    L.tile_least = tile_least(t, single);
    best = us;
  }
  const RowsGeom r = plan_rows(L.g, L.esize, sms, &us);
  if (r.rows > 0 && us < best) {
    L.plan = PLAN_ROWS;
    L.rows = r;
  }
}

// Steps of the next launch of n remaining steps: as many as the plan takes,
// without leaving a single step behind k_step_rows (4 = 2 + 2); 1 is a
// single-step launch where the plan's kernel takes no fewer than 2 (rows) or
// tile_least.  Forced steps take tiles down to one step.
inline int next_steps(const Lattice &L, long n, bool forced = false) {
  if (L.plan == PLAN_TILE)
    return n < L.tile_least && !forced ? 1 : (int)std::min<long>(n, L.tile.steps);
  if (L.plan == PLAN_ROWS) return n == 1 ? 1 : (n == 2 || n == 4 ? 2 : kRowSteps);
  return 1;
}

}  // namespace lbm
