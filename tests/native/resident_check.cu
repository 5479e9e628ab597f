// Host-compiled check of which resident batch members share an SM
// (lbm_internal.h, GB300's 228 KB of shared memory per SM and 1 KB reserved
// per block).  Built and run by tests/test_resident_cpu.py; prints "OK" and
// exits 0 when every check holds.
#include <stdio.h>

#include "../../paper_1107_4543_gb300/csrc/lbm_internal.h"

using namespace lbm;

int main() {
  const size_t sm = 228 * 1024, reserved = 1024, block = 227 * 1024;
  int failures = 0;
  for (int esize : {4, 2}) {
    long long last_pair = 0, last_resident = 0;
    for (long long n = 4; n < 8000; ++n) {
      const size_t smem = resident_smem(n, esize);
      // the planes and 26 (FP32) or PC_COUNT broadcast constants behind them
      const size_t table = (size_t)(esize == 4 ? (int)HL_COUNT : (int)PC_COUNT) * 8;
      if (smem < (size_t)9 * n * esize + table || smem % 16 != 0) ++failures;
      const bool resident = resident_bytes((int)n, 1, esize) <= block;
      const bool pair = resident_pairs(n, esize, sm, reserved);
      if (pair != (2 * smem + 2 * reserved <= sm)) ++failures;
      if (resident && smem > block) ++failures;      // alone it always fits
      if (resident) last_resident = n;
      if (resident && pair) last_pair = n;
      if (pair && last_pair != n && resident) ++failures;  // monotonic
      const ResidentKind kind = resident_kind(n, esize, sm, reserved);
      if (kind != (esize == 4 && n <= kResidentScalar ? RES_TINY : (pair ? RES_PAIRS : RES_ALONE)))
        ++failures;
    }
    printf("esize %d: pairs to %lld, resident to %lld\n", esize, last_pair, last_resident);
    if (esize == 4 && (last_pair != 3208 || last_resident != 3228)) ++failures;
    if (esize == 2 && (last_pair != 6421 || last_resident != 6456))
      ++failures;
  }
  if (failures) {
    printf("%d failures\n", failures);
    return 1;
  }
  printf("OK\n");
  return 0;
}
