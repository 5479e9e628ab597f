// Host-compiled check of the launches that take the last few steps of a
// lattice in tiles (plan.h): fewer than `least` steps go one by one, forced
// ones always in tiles, no launch takes more steps than its tiles hold, and
// `least` is where the estimates cross.  Built and run by
// tests/test_tile_rest_cpu.py; prints "OK" and exits 0 when every check holds.
#include <stdio.h>

#include "../../paper_1107_4543_gb300/csrc/plan.h"

using namespace lbm;

int main() {
  int failures = 0, tiles = 0, rests = 0;
  for (int esize : {4, 2})
    for (int nx : {2, 3, 5, 16, 53, 101, 256, 300, 512, 700, 3000})
      for (int ny : {2, 3, 16, 31, 101, 290, 512, 700, 3000}) {
        Lattice L;
        L.esize = esize;
        L.g = make_geom(nx, ny, esize == 4 ? 4 : 8, esize);
        plan_lattice(L, 152);
        if (L.plan != PLAN_TILE) continue;
        const TileGeom &t = L.tile;
        const int least = L.tile_least;
        const double single = single_us((double)nx * ny, esize);
        ++tiles;
        rests += least > 1;
        if (least < 1 || least > t.steps) ++failures;
        for (int n = 1; n < least; ++n)
          if (!(tile_us(t.by, n) > 1.25 * n * single)) ++failures;
        if (least < t.steps && tile_us(t.by, least) > 1.25 * least * single) ++failures;
        for (long n = 1; n <= 40; ++n) {
          long left = n;
          while (left > 0) {
            const int k = next_steps(L, left), f = next_steps(L, left, true);
            if (k != (left < least ? 1 : (int)(left < t.steps ? left : t.steps))) ++failures;
            if (f != (int)(left < t.steps ? left : t.steps)) ++failures;
            left -= k;
          }
        }
      }
  printf("%d lattices in tiles, %d with single last steps\n", tiles, rests);
  if (failures || tiles < 20 || rests < 5) {
    printf("%d failures\n", failures);
    return 1;
  }
  printf("OK\n");
  return 0;
}
