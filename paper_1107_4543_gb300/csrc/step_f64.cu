// Plain FP64 step: fused pull-stream + MRT collide on the full populations.
//
// The collision has the results of a plain matrix-vector implementation of
// section 2.1 (collide_f64), and this file is compiled with -fmad=false, so
// the step is bit-identical to a straightforward FP64 CPU implementation of
// the same definition.  Per node it moves 9 + 9 doubles (144 B) and performs
// ~119 FP64 operations; on GB300 the FP64 units (two lanes per clock and SM),
// not HBM, bound it.
#include "lbm_internal.h"
#include "node_xy.cuh"
#include "pdl.cuh"

namespace lbm {

// One node per thread and 32-thread blocks: whatever the size, the warps
// spread evenly over the SMs' FP64 units.  (Warp tasks of 64 nodes with
// 16-byte vectors, in 256-thread blocks, ran 64^2 on 16 of the 152 SMs, 19.9
// against 5.2 us per step, and 2048^2 at 951 against 917 - 946 us.)  A warp
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

// a / b correctly rounded (see Quotients)
__device__ __forceinline__ double quotient(double a, double b) {
  const Quotients Q(b, a, a, a);
  return Q.fast ? Q(a) : a / b;
}

// The step of a small lattice: four warps, one per scheduler of an SM, share
// the FP64 operations of 32 nodes, since one warp's 119 operations at 64
// cycles each are the time of a step while there are fewer warps than
// schedulers.  Three phases, 16 + 16 + 9 operations on the longest warp,
// exchange their sums, products and relaxed moments through shared memory;
// every value is formed by collide_f64's own operations, so the bits are
// the same.  164 operations in all: past two blocks per SM the plain form is
// the faster one.  us per step, plain / this: 64^2 5.1 / 3.1, 97 x 100 (304
// blocks, two per SM) 5.2 / 4.3, 101^2 (319) 5.2 / 5.6, 200^2 11.8 / 14.6.
__global__ void __launch_bounds__(128)
k_step_f64_split(const double *__restrict__ src, double *__restrict__ dst, Geom g, F64Params P) {
  enum { RHO, JX, JY, PXX, P3, P4, P5, P6, R7, R8, COUNT };
  __shared__ double sh[COUNT][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long n0 = blockIdx.x * 32LL + lane;
  const bool in = n0 < (long long)g.nx * g.ny;
  const long long n = in ? n0 : 0;
  int x, y;
  node_xy(n, g.nx, x, y);
  pdl_wait();
  double f[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    // a warp's own sums and outputs leave out what the others need
    if ((w == 1 && (i == 2 || i == 4)) || (w == 2 && (i == 0 || i == 1 || i == 3))) continue;
    int xs = x - CXd(i);
    xs = xs < 0 ? xs + g.nx : (xs >= g.nx ? xs - g.nx : xs);
    f[i] = __ldcg(src + (long long)i * g.plane + (long long)src_row(g, y, i) * g.rstride + xs);
  }
  double m = 0, k = 0;  // the moments a warp keeps for itself
  if (w == 0) {
    sh[RHO][lane] = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
    m = fma(2.0, fma(2.0, f[0], -f[1]) - f[2] - f[3] - f[4], f[5]) + f[6] + f[7] + f[8];
  } else if (w == 1) {
    const double d13 = f[1] - f[3];
    sh[JX][lane] = d13 + f[5] - f[6] - f[7] + f[8];
    m = fma(-2.0, d13, f[5]) - f[6] - f[7] + f[8];
  } else if (w == 2) {
    const double d24 = f[2] - f[4];
    sh[JY][lane] = d24 + f[5] + f[6] - f[7] - f[8];
    m = fma(-2.0, d24, f[5]) + f[6] - f[7] - f[8];
    k = f[5] - f[6] + f[7] - f[8];
  } else {
    m = fma(2.0, f[8], fma(2.0, f[7], fma(2.0, f[6], fma(2.0, f[5],
            fma(-4.0, f[0], -f[1]) - f[2] - f[3] - f[4]))));
    sh[PXX][lane] = f[1] - f[2] + f[3] - f[4];
  }
  __syncthreads();
  constexpr double c36 = 1.0 / 36.0, c12 = 1.0 / 12.0;
  const double rho = sh[RHO][lane], jx = sh[JX][lane], jy = sh[JY][lane];
  if (w == 0 || w == 3) {
    const double jxx = jx * jx, jyy = jy * jy;
    const double dj = quotient(3.0 * (jxx + jyy), rho);
    if (w == 0) sh[P4][lane] = c36 * (P.s4 * (m - (rho - dj)));
    else sh[P3][lane] = c36 * (P.s3 * (m - fma(-2.0, rho, dj)));
  } else if (w == 1) {
    const double jxx = jx * jx, jyy = jy * jy;
    sh[R7][lane] = P.s7 * (sh[PXX][lane] - quotient(jxx - jyy, rho));
    sh[P5][lane] = c12 * (P.s5 * (m + jx));
  } else {
    sh[R8][lane] = P.s8 * (k - quotient(jx * jy, rho));
    sh[P6][lane] = c12 * (P.s6 * (m + jy));
  }
  __syncthreads();
  const double p3 = sh[P3][lane], p4 = sh[P4][lane];
  auto put = [&](int i, double v) {
    if (in) dst[(long long)i * g.plane + (long long)y * g.rstride + x] = v;
  };
  if (w == 1) {
    const double p5 = sh[P5][lane], r7 = sh[R7][lane], t = fma(-2.0, p4, -p3);
    put(0, fma(-4.0, p4 - p3, f[0]));
    put(1, f[1] - fma(0.25, r7, fma(-2.0, p5, t)));
    put(3, f[3] - fma(0.25, r7, fma(2.0, p5, t)));
  } else if (w == 2) {
    const double p6 = sh[P6][lane], r7 = sh[R7][lane], t = fma(-2.0, p4, -p3);
    put(2, f[2] - fma(-0.25, r7, fma(-2.0, p6, t)));
    put(4, f[4] - fma(-0.25, r7, fma(2.0, p6, t)));
  } else {
    const double p5 = sh[P5][lane], p6 = sh[P6][lane], r8 = sh[R8][lane];
    const double u = fma(2.0, p3, p4);
    if (w == 0) {
      const double up = u + p5;
      put(5, f[5] - fma(0.25, r8, up + p6));
      put(8, f[8] - fma(-0.25, r8, up - p6));
    } else {
      const double um = u - p5;
      put(6, f[6] - fma(-0.25, r8, um + p6));
      put(7, f[7] - fma(0.25, r8, um - p6));
    }
  }
}

cudaError_t launch_step_f64(const Lattice &L, const void *src, void *dst, cudaStream_t st) {
  const long long n = (long long)L.g.nx * L.g.ny;
  if ((n + 31) / 32 <= 2LL * sm_count())  // see k_step_f64_split
    return launch_pdl(k_step_f64_split, (unsigned)((n + 31) / 32), 128, 0, st, (const double *)src,
                      (double *)dst, L.g, L.fp);
  return launch_pdl(k_step_f64, (unsigned)((n + 31) / 32), 32, 0, st, (const double *)src,
                    (double *)dst, L.g, L.fp);
}

}  // namespace lbm
