// Host-compiled check of how a lattice's steps are split into launches
// (plan.h): strips and tiles cover every node once and fit the limits of
// their kernels, and next_steps takes every step exactly once.  Built and
// run by tests/test_plan_cpu.py; prints "OK" and exits 0 when every check
// holds.
#include <stdio.h>
#include <stdlib.h>

#include <vector>

#include "../../paper_1107_4543_gb300/csrc/plan.h"

using namespace lbm;

static int failures = 0;
#define CHECK(cond, ...)                                  \
  do {                                                    \
    if (!(cond)) {                                        \
      if (failures < 20) {                                \
        printf("FAIL %s:%d: ", __FILE__, __LINE__);       \
        printf(__VA_ARGS__);                              \
        printf("\n");                                     \
      }                                                   \
      ++failures;                                         \
    }                                                     \
  } while (0)

static void check(int nx, int ny, int dtype, int esize) {
  const int V = vec_nodes(dtype), sms = 152;
  Lattice L;
  L.dtype = dtype;
  L.esize = esize;
  L.V = V;
  L.g = make_geom(nx, ny, V, esize);
  plan_lattice(L, sms);
  // rows: every chunk of every row is some task's own exactly once (its lanes
  // but `halo` on each side), for small lattices by enumeration
  for (int rows : {1, 8, 32}) {
    const RowsGeom r = rows_geom(L.g, rows);
    CHECK(r.rows >= 1 && r.segs >= 1 && (long long)r.segs * r.rows >= ny &&
              (long long)(r.segs - 1) * r.rows < ny,
          "segs %d x %d of %d rows", r.segs, r.rows, ny);
    const int per = rows_chunks(L.g) + 2 * r.halo;
    // a halo lane of the partial last chunk alone must hold a node per step
    CHECK(r.halo == 2 || nx % kRowsV == 0 || nx % kRowsV >= kRowSteps, "halo %d nx %d", r.halo, nx);
    if ((long long)nx * ny > 20000) continue;
    std::vector<int> seen((size_t)r.segs * per, 0);
    for (int t = 0; t < r.tasks; ++t)
      for (int lane = r.halo; lane < 32 - r.halo; ++lane) {
        const long long p = (32LL - 2 * r.halo) * t + lane;
        if (p < (long long)seen.size()) seen[(size_t)p]++;
      }
    for (size_t p = 0; p < seen.size(); ++p) {
      const int c = (int)(p % per) - r.halo;
      CHECK((c < 0 || c >= rows_chunks(L.g)) ? seen[p] <= 1 : seen[p] == 1, "position %zu seen %d", p,
            seen[p]);
    }
  }
  double rus = 0;
  const RowsGeom r = plan_rows(L.g, esize, sms, &rus);
  CHECK(rows_fit(L.g) ? (r.rows >= 1 && r.rows <= 48 && rus > 0) : r.rows == 0, "rows %d", r.rows);
  double us = 0;
  const TileGeom t = plan_tile(L.g, esize, sms, &us);
  if (t.steps > 0) {
    CHECK(t.steps <= kMaxTileSteps && t.ntx * t.nty <= sms, "tile %d %d %d", t.steps, t.ntx, t.nty);
    CHECK(t.bx % 2 == 0 && t.bx + 2 * tile_halo_x(t.steps) <= kTileCols, "bx %d steps %d", t.bx,
          t.steps);
    CHECK(tile_bytes(t.by, t.steps, esize) <= (size_t)kMaxSmem, "smem %d %d", t.by, t.steps);
    CHECK((long long)t.ntx * t.bx >= nx && (long long)(t.ntx - 1) * t.bx < nx, "ntx nx %d", nx);
    CHECK((long long)t.nty * t.by >= ny && (long long)(t.nty - 1) * t.by < ny, "nty ny %d", ny);
    // the last pair of an odd row fits the padding
    CHECK(nx % 2 == 0 || L.g.pitch > nx, "pitch %d nx %d", L.g.pitch, nx);
  }
  CHECK(L.plan != PLAN_TILE || L.tile.steps > 1, "tile plan of %d steps", L.tile.steps);
  for (long n = 1; n < 40; ++n) {
    long left = n;
    while (left > 0) {
      const int k = next_steps(L, left);
      CHECK(k >= 1 && k <= left, "next_steps %d of %ld", k, left);
      if (L.plan == PLAN_ROWS)
        CHECK(k == 2 || k == kRowSteps || (n == 1 && k == 1), "rows %d of %ld", k, n);
      left -= k;
    }
  }
}

int main() {
  for (int dtype : {LBM_F32DEV, LBM_F16DEV, LBM_BF16DEV}) {
    const int esize = dtype == LBM_F32DEV ? 4 : 2;
    for (int nx : {2, 3, 4, 5, 7, 8, 9, 31, 64, 101, 119, 121, 240, 241, 512, 700, 1000, 1024, 1500,
                   4097, 8192, 20000})
      for (int ny : {2, 3, 5, 8, 16, 23, 101, 512, 777, 1111, 3071, 8192}) check(nx, ny, dtype, esize);
  }
  // the lattices with which the GPU tests reach k_step_rows
  auto rows_plan = [](int nx, int ny, int dtype) {
    Lattice L;
    L.dtype = dtype;
    L.esize = dtype == LBM_F32DEV ? 4 : 2;
    L.V = vec_nodes(dtype);
    L.g = make_geom(nx, ny, L.V, L.esize);
    plan_lattice(L, 152);
    CHECK(L.plan == PLAN_ROWS, "plan of %d x %d: %d", nx, ny, (int)L.plan);
  };
  for (int k = 0; k < 4; ++k) rows_plan(1200 + k, 1101, LBM_F32DEV);
  rows_plan(700001, 2, LBM_F32DEV);
  rows_plan(420003, 3, LBM_F32DEV);
  for (int k = 0; k < 8; ++k) rows_plan(2496 + k, 2101, LBM_F16DEV);
  rows_plan(2501, 2101, LBM_BF16DEV);
  // the FP64 types step one by one
  for (int dtype : {LBM_F64, LBM_F64DEV}) {
    Lattice L;
    L.dtype = dtype;
    L.esize = 8;
    L.g = make_geom(64, 64, 2, 8);
    plan_lattice(L, 152);
    CHECK(L.plan == PLAN_SINGLE && next_steps(L, 10) == 1, "FP64 plan");
  }
  if (failures) {
    printf("%d failures\n", failures);
    return 1;
  }
  printf("OK\n");
  return 0;
}
