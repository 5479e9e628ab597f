// Field I/O kernels of the deviation storage types (FP32, FP16, BF16):
// equilibrium initialisation from device fields, the largest deviation that
// sets the FP16 storage scale, and the moments.  The FP64 storage type keeps
// the canonical kernels of aux.cu (bit parity with a plain FP64 version).
//
// The equilibrium of section 2.3, f^eq = M^-1 m^eq, equals the second-order
// polynomial  w_i [rho + 3 c_i.j + 9/2 (c_i.j)^2 / rho - 3/2 |j|^2 / rho]
// with weights 4/9, 1/9 (axis) and 1/36 (diagonal).  What is stored is the
// deviation f^eq(rho, j) - f^eq(rho0, j0), formed here from the differences
// rho - rho0, j - j0, jx^2/rho - jx0^2/rho0, jy^2/rho - jy0^2/rho0 and
// jx jy/rho - jx0 jy0/rho0: every term is of the size of the perturbation,
// so nothing of order one is subtracted after rounding.  GB300's FP64 rate
// (1/64 of FP32) bounded these kernels, not their 60 bytes per node (8192^2
// FP32: init 6.1 ms, moments 4.6 ms, against 0.6 ms of HBM traffic), so only
// what needs FP64 runs there: the init forms the six differences in FP64 and
// their linear combinations as float-float sums (feq_rounded), and the
// moments sum the stored values as float-float where those sums are exact
// (sums_exact): 1.4 and 2.5 ms, with the FP64 form's bits in both.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include "bounds.cuh"
#include "lbm_internal.h"
#include "node_xy.cuh"

namespace lbm {
namespace {

// reference state and its quadratic terms (host-computed)
struct RefState {
  double rho0, jx0, jy0;
  double axx0, ayy0, axy0;  // jx0^2/rho0, jy0^2/rho0, jx0 jy0/rho0
};

RefState make_ref(const AuxView &a) {
  RefState r;
  r.rho0 = a.rho0;
  r.jx0 = a.jx0;
  r.jy0 = a.jy0;
  r.axx0 = a.jx0 * a.jx0 / a.rho0;
  r.ayy0 = a.jy0 * a.jy0 / a.rho0;
  r.axy0 = a.jx0 * a.jy0 / a.rho0;
  return r;
}

__device__ __forceinline__ int wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// rho <= 0 or a value that is not finite, from the bits
__device__ __forceinline__ bool field_bad(double r, double u, double v) {
  auto top = [](double d) { return ((unsigned)__double2hiint(d) >> 20) & 0x7ffu; };
  const bool zero = (((unsigned)__double2hiint(r) << 1) | (unsigned)__double2loint(r)) == 0u;
  return zero || __double2hiint(r) < 0 || top(r) == 0x7ffu || top(u) == 0x7ffu || top(v) == 0x7ffu;
}

// f^eq_i(rho, rho u) - f^eq_i(rho0, j0), i = 0..8
__device__ __forceinline__ void feq_deviation(const RefState &R, double r, double u, double v,
                                              double d[9]) {
  const double jx = r * u, jy = r * v;
  const double dr = r - R.rho0;
  const double ex = 3.0 * (jx - R.jx0), ey = 3.0 * (jy - R.jy0);
  // jx^2 / rho = rho u^2 etc.: the fields give u, so no division is needed
  // (GB300's FP64 divide is the costliest step of this FP64-bound kernel)
  const double A = jx * u - R.axx0;
  const double B = jy * v - R.ayy0;
  const double C = jx * v - R.axy0;
  const double t1 = dr + 3.0 * A - 1.5 * B;  // axis x: 9/2 A - 3/2 (A + B)
  const double t2 = dr + 3.0 * B - 1.5 * A;  // axis y
  const double t5 = dr + 3.0 * (A + B);      // diagonals: 9/2 (A + B +- 2C) - 3/2 (A + B)
  const double p = t5 + 9.0 * C, q = t5 - 9.0 * C;
  constexpr double w0 = 4.0 / 9.0, w1 = 1.0 / 9.0, w5 = 1.0 / 36.0;
  d[0] = w0 * (dr - 1.5 * (A + B));
  d[1] = w1 * (t1 + ex);
  d[2] = w1 * (t2 + ey);
  d[3] = w1 * (t1 - ex);
  d[4] = w1 * (t2 - ey);
  d[5] = w5 * (p + ex + ey);
  d[6] = w5 * (q - ex + ey);
  d[7] = w5 * (p - ex - ey);
  d[8] = w5 * (q + ex - ey);
}

// float-float: an unevaluated sum h + l of ~48 bits
struct FF {
  float h, l;
};
// s + e = a + b exactly (Knuth's TwoSum; additions alone, so no contraction
// into multiply-adds can touch it)
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  e += a.l + b.l;
  const float h = s + e;  // |s| >= |e|: the quick form of TwoSum is exact
  return {h, e - (h - s)};
}
__device__ __forceinline__ FF ff_neg(FF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ FF ff_scale(FF a, float p2) { return {a.h * p2, a.l * p2}; }  // p2 = 2^k
// a (wh + wl)
__device__ __forceinline__ FF ff_mul(FF a, float wh, float wl) {
  const float p = __fmul_rn(a.h, wh);
  float e = __fmaf_rn(a.h, wh, -p);
  e = __fmaf_rn(a.h, wl, __fmaf_rn(a.l, wh, e));
  const float h = p + e;
  return {h, e - (h - p)};
}
// d as float-float from its bits (conversions run at the FP64 rate): the top
// 24 significand bits, then the low 29 as a scaled integer.  Values below
// 2^-74 read as zero and add that much to `lost`; false for |d| >= 2^100,
// infinities and NaN.
__device__ __forceinline__ bool ff_split(double d, FF &o, float &lost) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned mag = hi & 0x7fffffffu, sign = hi & 0x80000000u, e = mag >> 20;
  if (e < 949u) {
    o = {0.0f, 0.0f};
    lost += (mag | lo) != 0u ? 5.3e-23f : 0.0f;  // 2^-74
    return true;
  }
  o.h = __uint_as_float(sign | (__funnelshift_l(lo, mag, 3) - (896u << 23)));
  const float unit = __uint_as_float(sign | ((e - 948u) << 23));  // 2^(e - 1023 - 52)
  o.l = (float)(int)(lo & 0x1fffffffu) * unit;
  return e < 1123u;
}

// The nine deviations of feq_deviation rounded to FP32, exactly as the FP64
// form rounds them: the six O(perturbation) differences in FP64 with the
// same operations, their combinations as float-float to ~2^-44 of the
// largest term (in units of the diagonal weight 1/36: the other weights are
// 4 and 16 times that).  A value whose rounding that error could change --
// one node in several thousand -- or a difference outside the split's range returns false,
// and the caller takes the FP64 form.
__device__ __forceinline__ bool feq_rounded(const RefState &R, double r, double u, double v,
                                            float d[9]) {
  const double jx = r * u, jy = r * v;
  constexpr double W36 = 1.0 / 36.0, W12 = 1.0 / 12.0, W24 = 1.0 / 24.0;
  constexpr float w36h = (float)W36, w36l = (float)(W36 - (double)w36h);
  constexpr float w12h = (float)W12, w12l = (float)(W12 - (double)w12h);
  constexpr float w24h = (float)W24, w24l = (float)(W24 - (double)w24h);
  FF t[6];
  float lost = 0.0f;
  bool ok = ff_split(r - R.rho0, t[0], lost);
  ok &= ff_split(jx - R.jx0, t[1], lost);
  ok &= ff_split(jy - R.jy0, t[2], lost);
  ok &= ff_split(fma(jx, u, -R.axx0), t[3], lost);
  ok &= ff_split(fma(jy, v, -R.ayy0), t[4], lost);
  ok &= ff_split(fma(jx, v, -R.axy0), t[5], lost);
  const FF dr = ff_mul(t[0], w36h, w36l);
  const FF X = ff_mul(t[1], w12h, w12l), Y = ff_mul(t[2], w12h, w12l);
  const FF a = ff_mul(t[3], w24h, w24l), b = ff_mul(t[4], w24h, w24l);
  const FF c = ff_scale(t[5], 0.25f);
  const FF S = ff_add(a, b);
  const FF t1 = ff_add(ff_add(dr, ff_neg(b)), ff_scale(a, 2.0f));
  const FF t2 = ff_add(ff_add(dr, ff_neg(a)), ff_scale(b, 2.0f));
  const FF t5 = ff_add(dr, ff_scale(S, 2.0f));
  const FF p = ff_add(t5, c), q = ff_add(t5, ff_neg(c));
  const FF xy = ff_add(X, Y), yx = ff_add(Y, ff_neg(X));
  const FF o[9] = {ff_add(dr, ff_neg(S)), ff_add(t1, X),           ff_add(t2, Y),
                   ff_add(t1, ff_neg(X)), ff_add(t2, ff_neg(Y)),   ff_add(p, xy),
                   ff_add(q, yx),         ff_add(p, ff_neg(xy)),   ff_add(q, ff_neg(yx))};
  // 2^-43 of the terms' magnitudes (the rest population has no term linear
  // in the velocity, which is the largest elsewhere), and what the split
  // dropped
  const float tol0 = 1.14e-13f * (fabsf(dr.h) + 4.0f * (fabsf(a.h) + fabsf(b.h)) + fabsf(c.h)) +
                     lost;
  const float tol = tol0 + 1.14e-13f * (fabsf(X.h) + fabsf(Y.h));
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const float t = i == 0 ? tol0 : tol;
    ok &= o[i].h + (o[i].l + t) == o[i].h && o[i].h + (o[i].l - t) == o[i].h;
    d[i] = o[i].h * (i == 0 ? 16.0f : (i <= 4 ? 4.0f : 1.0f));
  }
  return ok;
}

// feq_rounded, or the FP64 form where it cannot tell
__device__ __forceinline__ void feq_f32(const RefState &R, double r, double u, double v,
                                        float f[9]) {
  if (feq_rounded(R, r, u, v, f)) return;
  double d[9];
  feq_deviation(R, r, u, v, d);
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = (float)d[i];
}

// storage of an FP32 deviation (FP16: times the power-of-two scale, exact)
template <typename T>
__device__ __forceinline__ T encode_f32(float d, float scale);
template <>
__device__ __forceinline__ float encode_f32<float>(float d, float) {
  return d;
}
template <>
__device__ __forceinline__ __half encode_f32<__half>(float d, float scale) {
  return __float2half_rn(d * scale);
}
template <>
__device__ __forceinline__ __nv_bfloat16 encode_f32<__nv_bfloat16>(float d, float) {
  return __float2bfloat16_rn(d);
}

// Population i of node x goes to slot x - c_i, where the next step's pull
// (f_i(x) = P_i(x - c_i)) reads it.  bad counts nodes whose field is not
// finite or has rho <= 0.
// one node of the equilibrium init: the deviations of f^eq(r, (u, v)) into
// the slots the next pull reads; returns whether the field is invalid
template <typename T>
__device__ __forceinline__ bool init_node(const AuxView &a, const RefState &R, int x, int y,
                                          double r, double u, double v) {
  T *buf = static_cast<T *>(a.buf);
  T e[9];
  if constexpr (sizeof(T) == 8) {
    feq_deviation(R, r, u, v, e);
  } else {
    float f[9];
    feq_f32(R, r, u, v, f);
    const float scale = (float)a.scale;
#pragma unroll
    for (int i = 0; i < 9; ++i) e[i] = encode_f32<T>(f[i], scale);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int xs = wrap(x - CXd(i), a.g.nx), ys = wrap(y - CYd(i), a.g.nyw);
    buf[(long long)i * a.g.plane + (long long)ys * a.g.rstride + xs] = e[i];
  }
  return field_bad(r, u, v);
}

template <typename T>
__global__ void __launch_bounds__(256) k_init_dev(AuxView a, RefState R, const double *rho,
                                                  const double *ux, const double *uy,
                                                  unsigned int *bad) {
  const int nx = a.g.nx, ny = a.g.ny;
  const long long N = (long long)nx * ny;
  unsigned int nbad = 0;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int x, y;
    node_xy(n, nx, x, y);
    if (init_node<T>(a, R, x, y, rho[n], ux[n], uy[n])) ++nbad;
  }
  if (bad && nbad) atomicAdd(bad, nbad);
}

__global__ void __launch_bounds__(256) k_maxdev_dev(AuxView a, RefState R, const double *rho,
                                                    const double *ux, const double *uy,
                                                    unsigned int *max_bits) {
  const long long N = (long long)a.g.nx * a.g.ny;
  float m = 0.0f;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    float d[9];
    feq_f32(R, rho[n], ux[n], uy[n], d);
#pragma unroll
    for (int i = 0; i < 9; ++i) m = fmaxf(m, fabsf(d[i]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(max_bits, __float_as_uint(m));
}

template <typename T>
__device__ __forceinline__ float decode_f32(T s, float inv_scale);
template <>
__device__ __forceinline__ float decode_f32<float>(float s, float) {
  return s;
}
template <>
__device__ __forceinline__ float decode_f32<__half>(__half s, float inv_scale) {
  return __half2float(s) * inv_scale;  // a power of two
}
template <>
__device__ __forceinline__ float decode_f32<__nv_bfloat16>(__nv_bfloat16 s, float) {
  return __bfloat162float(s);
}

__device__ __forceinline__ void ff_acc(FF &s, float a) {
  float e;
  two_sum(s.h, a, s.h, e);
  s.l += e;
}
// a float's double by its bits (conversions run at the FP64 rate)
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), mag = b & 0x7fffffffu, e = mag >> 23;
  if (e - 1u >= 254u && mag != 0u) return (double)f;  // subnormal, infinite, NaN
  const unsigned hi = mag == 0u ? 0u : (mag >> 3) + 0x38000000u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(mag << 29));
}
__device__ __forceinline__ double ff_value(FF s) { return widen(s.h) + widen(s.l); }
// Whether the sums over nine FP32 values come out exact both in FP64 and as
// float-float, so that the cheaper one gives the FP64 form's bits.  Values of
// exponents e0 .. e1 (zeros apart) are multiples of 2^(e0 - 23), and partial
// sums stay below 2^(e1 + 5): FP64 holds them for e1 - e0 <= 25, and the FP32
// sum of the two_sum errors, each at most 2^(e1 - 20), for e1 - e0 <= 18.
// Infinities, NaN and sums that FP32 could not hold fail the test too.
__device__ __forceinline__ bool sums_exact(const float (&f)[9]) {
  unsigned top = 0u, low = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const unsigned mag = __float_as_uint(f[i]) & 0x7fffffffu;
    top = max(top, mag);
    low = min(low, mag - 1u);  // a zero is no bound
  }
  top >>= 23;
  return top - ((low + 1u) >> 23) <= 18u && top <= 248u;
}

// rho = rho0 + sum f', j = j0 + sum c f' of the pre-collision populations
// f_i(x) = P_i(x - c_i); u = j / rho
// rho, u of node (x, y) from its pre-collision populations
template <typename T>
__device__ __forceinline__ void moments_node(const AuxView &a, int x, int y, float inv_scale,
                                             double &r, double &u, double &v) {
  const T *buf = static_cast<const T *>(a.buf);
  if constexpr (sizeof(T) == 8) {
    double f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int xs = wrap(x - CXd(i), a.g.nx), ys = wrap(y - CYd(i), a.g.nyw);
      f[i] = buf[(long long)i * a.g.plane + (long long)ys * a.g.rstride + xs];
    }
    r = a.rho0 + (f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8]);
    const double jx = a.jx0 + (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]);
    const double jy = a.jy0 + (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]);
    const double inv = 1.0 / r;
    u = jx * inv;
    v = jy * inv;
  } else {
    // the FP64 sums from left to right; as float-float and one FP64 addition
    // where that is known to give the same
    float f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int xs = wrap(x - CXd(i), a.g.nx), ys = wrap(y - CYd(i), a.g.nyw);
      f[i] = decode_f32<T>(buf[(long long)i * a.g.plane + (long long)ys * a.g.rstride + xs],
                           inv_scale);
    }
    double S0, S1, S2;
    if (sums_exact(f)) {
      FF s0{f[0], 0.0f}, s1{f[1], 0.0f}, s2{f[2], 0.0f};
#pragma unroll
      for (int i = 1; i < 9; ++i) ff_acc(s0, f[i]);
      ff_acc(s1, -f[3]); ff_acc(s1, f[5]); ff_acc(s1, -f[6]); ff_acc(s1, -f[7]); ff_acc(s1, f[8]);
      ff_acc(s2, -f[4]); ff_acc(s2, f[5]); ff_acc(s2, f[6]); ff_acc(s2, -f[7]); ff_acc(s2, -f[8]);
      S0 = ff_value(s0);
      S1 = ff_value(s1);
      S2 = ff_value(s2);
    } else {
      double d[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) d[i] = (double)f[i];
      S0 = d[0] + d[1] + d[2] + d[3] + d[4] + d[5] + d[6] + d[7] + d[8];
      S1 = d[1] - d[3] + d[5] - d[6] - d[7] + d[8];
      S2 = d[2] - d[4] + d[5] + d[6] - d[7] - d[8];
    }
    r = a.rho0 + S0;
    const double jx = a.jx0 + S1, jy = a.jy0 + S2;
    const double inv = recip_rounds(r) ? recip(r) : 1.0 / r;
    u = jx * inv;
    v = jy * inv;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_moments_dev(AuxView a, double *rho, double *ux,
                                                     double *uy) {
  const int nx = a.g.nx, ny = a.g.ny;
  const long long N = (long long)nx * ny;
  const float inv_scale = (float)(1.0 / a.scale);  // a power of two
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int x, y;
    node_xy(n, nx, x, y);
    moments_node<T>(a, x, y, inv_scale, rho[n], ux[n], uy[n]);
  }
}

// Batched forms: block b covers nodes [start, start + count) of member
// blocks[b].member, whose fields sit at poff[member] of the packed arrays
// (rho at `stage`, ux at stage + total, uy at stage + 2 total).  The
// per-node arithmetic is that of the single-lattice kernels.
__device__ __forceinline__ RefState ref_of(const AuxView &a) {
  RefState r;
  r.rho0 = a.rho0;
  r.jx0 = a.jx0;
  r.jy0 = a.jy0;
  r.axx0 = a.jx0 * a.jx0 / a.rho0;
  r.ayy0 = a.jy0 * a.jy0 / a.rho0;
  r.axy0 = a.jx0 * a.jy0 / a.rho0;
  return r;
}

template <typename T>
__device__ __forceinline__ void batch_init_block(const AuxView &a, const IoBlock &B,
                                                 const double *r_, const double *u_,
                                                 const double *v_, unsigned int *bad) {
  const RefState R = ref_of(a);
  unsigned int nbad = 0;
  for (int j = threadIdx.x; j < B.count; j += blockDim.x) {
    const long long n = B.start + j;
    int x, y;
    node_xy(n, a.g.nx, x, y);
    if (init_node<T>(a, R, x, y, r_[n], u_[n], v_[n])) ++nbad;
  }
  if (nbad) atomicAdd(bad + B.member, nbad);
}

__global__ void __launch_bounds__(256) k_batch_init_dev(const AuxView *__restrict__ views,
                                                        const IoBlock *__restrict__ blocks,
                                                        const long long *__restrict__ poff,
                                                        long long total, const double *stage,
                                                        unsigned int *bad, int members) {
  const IoBlock B = blocks[blockIdx.x];
  if (!bounds::ok(B.member >= 0 && B.member < members, bounds::IO_BLOCK)) return;
  if (!bounds::ok(B.start >= 0 && B.count >= 0 &&
                      B.start + B.count <= (long long)views[B.member].g.nx * views[B.member].g.ny &&
                      poff[B.member] + B.start + B.count <= total,
                  bounds::IO_BLOCK))
    return;
  const AuxView &a = views[B.member];
  const double *r = stage + poff[B.member];
  switch (a.dtype) {
    case LBM_F32DEV: batch_init_block<float>(a, B, r, r + total, r + 2 * total, bad); break;
    case LBM_F16DEV: batch_init_block<__half>(a, B, r, r + total, r + 2 * total, bad); break;
    default: batch_init_block<__nv_bfloat16>(a, B, r, r + total, r + 2 * total, bad); break;
  }
}

template <typename T>
__device__ __forceinline__ void batch_moments_block(const AuxView &a, const IoBlock &B,
                                                    double *r_, double *u_, double *v_) {
  const float inv_scale = (float)(1.0 / a.scale);  // a power of two
  for (int j = threadIdx.x; j < B.count; j += blockDim.x) {
    const long long n = B.start + j;
    int x, y;
    node_xy(n, a.g.nx, x, y);
    moments_node<T>(a, x, y, inv_scale, r_[n], u_[n], v_[n]);
  }
}

__global__ void __launch_bounds__(256) k_batch_moments_dev(const AuxView *__restrict__ views,
                                                           const IoBlock *__restrict__ blocks,
                                                           const long long *__restrict__ poff,
                                                           long long total, double *stage,
                                                           int members) {
  const IoBlock B = blocks[blockIdx.x];
  if (!bounds::ok(B.member >= 0 && B.member < members, bounds::IO_BLOCK)) return;
  if (!bounds::ok(B.start >= 0 && B.count >= 0 &&
                      B.start + B.count <= (long long)views[B.member].g.nx * views[B.member].g.ny &&
                      poff[B.member] + B.start + B.count <= total,
                  bounds::IO_BLOCK))
    return;
  const AuxView &a = views[B.member];
  double *r = stage + poff[B.member];
  switch (a.dtype) {
    case LBM_F32DEV: batch_moments_block<float>(a, B, r, r + total, r + 2 * total); break;
    case LBM_F16DEV: batch_moments_block<__half>(a, B, r, r + total, r + 2 * total); break;
    default: batch_moments_block<__nv_bfloat16>(a, B, r, r + total, r + 2 * total); break;
  }
}

unsigned grid_for(long long n) {
  long long g = (n + 255) / 256;
  long long cap = (long long)sm_count() * 16;
  return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

__global__ void __launch_bounds__(256) k_batch_maxdev_fp16(const AuxView *__restrict__ views,
                                                           const IoBlock *__restrict__ blocks,
                                                           const long long *__restrict__ poff,
                                                           long long total, const double *stage,
                                                           unsigned int *max_bits, int members) {
  const IoBlock B = blocks[blockIdx.x];
  if (!bounds::ok(B.member >= 0 && B.member < members, bounds::IO_BLOCK)) return;
  if (!bounds::ok(B.start >= 0 && B.count >= 0 &&
                      B.start + B.count <= (long long)views[B.member].g.nx * views[B.member].g.ny &&
                      poff[B.member] + B.start + B.count <= total,
                  bounds::IO_BLOCK))
    return;
  const AuxView &a = views[B.member];
  if (a.dtype != LBM_F16DEV) return;  // block-uniform
  const RefState R = ref_of(a);
  const double *r = stage + poff[B.member];
  float m = 0.0f;
  for (int j = threadIdx.x; j < B.count; j += blockDim.x) {
    const long long n = B.start + j;
    float d[9];
    feq_f32(R, r[n], r[total + n], r[2 * total + n], d);
#pragma unroll
    for (int i = 0; i < 9; ++i) m = fmaxf(m, fabsf(d[i]));
  }
  // one atomic per block (a member's blocks all update the same word)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float wmax[8];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, wmax[w]);
    atomicMax(max_bits + B.member, __float_as_uint(m));
  }
}

__global__ void k_batch_set_scales(AuxView *views0, AuxView *views1, BatchEntry *const *ent,
                                   const unsigned int *max_bits, const double *floor_,
                                   double *scale_out, int members) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= members || views0[k].dtype != LBM_F16DEV || ent[k] == nullptr) return;
  const double m = fmax((double)__uint_as_float(max_bits[k]), floor_[k]);
  const double s = fp16_scale(m);
  views0[k].scale = s;
  views1[k].scale = s;
  ent[k]->dp.scale = (float)s;
  ent[k]->dp.inv_scale = (float)(1.0 / s);
  scale_out[k] = s;
}

}  // namespace

cudaError_t launch_init_dev(const AuxView &a, const double *rho, const double *ux,
                            const double *uy, cudaStream_t st, unsigned int *bad) {
  const long long N = (long long)a.g.nx * a.g.ny;
  if (bad) {
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
  }
  const RefState R = make_ref(a);
  const unsigned grid = grid_for(N);
  switch (a.dtype) {
    case LBM_F32DEV: k_init_dev<float><<<grid, 256, 0, st>>>(a, R, rho, ux, uy, bad); break;
    case LBM_F16DEV: k_init_dev<__half><<<grid, 256, 0, st>>>(a, R, rho, ux, uy, bad); break;
    case LBM_BF16DEV:
      k_init_dev<__nv_bfloat16><<<grid, 256, 0, st>>>(a, R, rho, ux, uy, bad);
      break;
    case LBM_F64DEV: k_init_dev<double><<<grid, 256, 0, st>>>(a, R, rho, ux, uy, bad); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_maxdev_dev(const AuxView &a, const double *rho, const double *ux,
                              const double *uy, unsigned int *max_bits, cudaStream_t st) {
  const long long N = (long long)a.g.nx * a.g.ny;
  cudaError_t e = cudaMemsetAsync(max_bits, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  k_maxdev_dev<<<grid_for(N), 256, 0, st>>>(a, make_ref(a), rho, ux, uy, max_bits);
  return cudaGetLastError();
}

cudaError_t launch_batch_fp16_scales(AuxView *views0, AuxView *views1, BatchEntry *const *ent,
                                     const IoBlock *blocks, long long nblocks,
                                     const long long *poff, long long total, const double *stage,
                                     unsigned int *max_bits, const double *floor_,
                                     double *scale_out, int members, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(max_bits, 0, sizeof(unsigned int) * members, st);
  if (e != cudaSuccess) return e;
  if (nblocks > 0)
    k_batch_maxdev_fp16<<<(unsigned)nblocks, 256, 0, st>>>(views0, blocks, poff, total, stage,
                                                           max_bits, members);
  k_batch_set_scales<<<(members + 127) / 128, 128, 0, st>>>(views0, views1, ent, max_bits, floor_,
                                                            scale_out, members);
  return cudaGetLastError();
}

cudaError_t launch_batch_init_dev(const AuxView *views, const IoBlock *blocks, long long nblocks,
                                  const long long *poff, long long total, const double *stage,
                                  unsigned int *bad, int members, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(unsigned int) * members, st);
  if (e != cudaSuccess || nblocks < 1) return e;
  k_batch_init_dev<<<(unsigned)nblocks, 256, 0, st>>>(views, blocks, poff, total, stage, bad,
                                                      members);
  return cudaGetLastError();
}

cudaError_t launch_batch_moments_dev(const AuxView *views, const IoBlock *blocks,
                                     long long nblocks, const long long *poff, long long total,
                                     double *stage, int members, cudaStream_t st) {
  if (nblocks < 1) return cudaSuccess;
  k_batch_moments_dev<<<(unsigned)nblocks, 256, 0, st>>>(views, blocks, poff, total, stage,
                                                         members);
  return cudaGetLastError();
}

cudaError_t launch_moments_dev(const AuxView &a, double *rho, double *ux, double *uy,
                               cudaStream_t st) {
  const long long N = (long long)a.g.nx * a.g.ny;
  const unsigned grid = grid_for(N);
  switch (a.dtype) {
    case LBM_F32DEV: k_moments_dev<float><<<grid, 256, 0, st>>>(a, rho, ux, uy); break;
    case LBM_F16DEV: k_moments_dev<__half><<<grid, 256, 0, st>>>(a, rho, ux, uy); break;
    case LBM_BF16DEV: k_moments_dev<__nv_bfloat16><<<grid, 256, 0, st>>>(a, rho, ux, uy); break;
    case LBM_F64DEV: k_moments_dev<double><<<grid, 256, 0, st>>>(a, rho, ux, uy); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Debug-build self-test of the index checks: one checked access with an
// index past its bound, which the check turns into index 0 of a one-element
// array (so nothing outside it is touched) while setting the SELFTEST bit.
__global__ void k_bounds_selftest(unsigned int *one) {
  const int i = bounds::ck(threadIdx.x + 1, 1, bounds::SELFTEST);
  one[i] = 1u;
}

cudaError_t launch_bounds_selftest(unsigned int *one, cudaStream_t st) {
  k_bounds_selftest<<<1, 1, 0, st>>>(one);
  return cudaGetLastError();
}

unsigned bounds_word_io(bool reset) { return bounds::read_word(reset); }

}  // namespace lbm
