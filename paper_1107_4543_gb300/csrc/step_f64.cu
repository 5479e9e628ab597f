// Plain FP64 step: fused pull-stream + MRT collide on the full populations.
//
// The collision has the results of a plain matrix-vector implementation of
// section 2.1 (collide_f64), and this file is compiled with -fmad=false, so
// the step is bit-identical to a straightforward FP64 CPU implementation of
// the same definition.  Per node it moves 9 + 9 doubles (144 B) and performs
// ~118 FP64 operations; on GB300 the FP64 units (two lanes per clock and SM),
// not HBM, bound it.
#include "lbm_internal.h"
#include "node_xy.cuh"
#include "pdl.cuh"

namespace lbm {

// One node per thread and 32-thread blocks: whatever the size, the warps
// spread evenly over the SMs' FP64 units.  (Warp tasks of 64 nodes with
// 16-byte vectors, in 256-thread blocks, ran 64^2 on 16 of the 152 SMs, 19.9
// against 5.2 us per step, and 2048^2 at 951 against 909 - 946 us.)  A warp
// instruction holds a scheduler's FP64 unit for 64 cycles however many lanes
// are active, so blocks of fewer nodes gain nothing (8 per warp: 64^2 at
// 5.9 us).
__global__ void __launch_bounds__(32)
k_step_f64(const double *__restrict__ src, double *__restrict__ dst, Geom g, F64Params P) {
  const long long n = blockIdx.x * 32LL + threadIdx.x;
  int x, y;
  node_xy(n, g.nx, x, y);
  pdl_wait();
  if (y >= g.ny) return;
  double f[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    int xs = x - CXd(i);
    xs = xs < 0 ? xs + g.nx : (xs >= g.nx ? xs - g.nx : xs);
    f[i] = __ldcg(src + (long long)i * g.plane + (long long)src_row(g, y, i) * g.rstride + xs);
  }
  collide_f64(f, P);
#pragma unroll
  for (int i = 0; i < 9; ++i) dst[(long long)i * g.plane + (long long)y * g.rstride + x] = f[i];
}

cudaError_t launch_step_f64(const Lattice &L, const void *src, void *dst, cudaStream_t st) {
  const long long n = (long long)L.g.nx * L.g.ny;
  return launch_pdl(k_step_f64, (unsigned)((n + 31) / 32), 32, 0, st, (const double *)src,
                    (double *)dst, L.g, L.fp);
}

}  // namespace lbm
