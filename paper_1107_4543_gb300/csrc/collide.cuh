// D2Q9 MRT collision at one node, in registers (device helpers).
//
// Moments m = M f with M the Lallemand-Luo D2Q9 matrix in the paper's row
// order rho, jx, jy, e, eps, qx, qy, pxx, pxy (section 2.1, Eq. q-macro);
// equilibrium moments of section 2.3; relaxation of the non-conserved
// moments with S = diag(0,0,0,s_e,s_eps,s_qx,s_qy,s_pxx,s_pxy) (section 2.1,
// Eq. eq_noconservative); back-transform f <- f - M^-1 S (m - m^eq) with
// M^-1 = M^T D^-1, D = diag(9,6,6,36,36,12,12,4,4) (M has orthogonal rows).
// The 9x9 transforms are unrolled by hand over the nonzero entries
// (0, +-1, +-2, +-4) and need no tensor cores.  Single steps of the 32- and
// 16-bit types are bound by HBM, several steps per launch by the FMA pipe, the
// FP64 types by the FP64 pipe.
#pragma once

namespace lbm {

// Rates pre-divided by the row norms D_k: k3 = s_e/36, k4 = s_eps/36,
// k5 = s_qx/12, k6 = s_qy/12, k7 = s_pxx/4, k8 = s_pxy/4.  Every constant
// that enters the FP32 collision is carried as an unevaluated FP32 sum
// hi + lo (accurate to ~2^-48): a systematic rounding of a constant does not
// average out but integrates over thousands of steps.  The optimized rates
// sit next to 2, where the physics lives in sigma = 1/s - 1/2 (10^-3 ..
// 10^-6); one FP32 rounding of s_e/36 already moves sigma_e by ~1e-5
// relative, a 1e-6 amplitude error after 2000 steps of a damped wave.
struct DevParams {
  float rho0, jx0, jy0;          // reference state (FP32-exact by construction)
  float k3, k4, k5, k6, k7, k8;  // s/D, high parts
  float l3, l4, l5, l6, l7, l8;  // s/D, low parts
  float q0h, q0l;                // |j0|^2
  float d0h, d0l;                // jx0^2 - jy0^2
  float x0h, x0l;                // jx0 jy0
  float i2h, i2l;                // 1 / rho0^2
  float scale, inv_scale;        // FP16 storage: stored = f' * scale
};

// a * (h + l) with the low part folded in by one FMA, or a * h alone when
// the low parts are not wanted
template <bool PRECISE>
__device__ __forceinline__ float mul_hl(float a, float h, float l) {
  return PRECISE ? fmaf(a, h, a * l) : a * h;
}

// 1 / d by the hardware reciprocal
__device__ __forceinline__ float rcp_approx(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}

// Deviation form: f' = f - f^eq(rho0, j0); the base carries the moments
// m^eq(rho0, j0), so rho = rho0 + rho', j = j0 + j' and the non-equilibrium
// parts are n = m' - [m^eq(rho, j) - m^eq(rho0, j0)].  Written so that FP32
// rounding never acts on a large quantity that then cancels:
//   * each n_k is formed directly from partial sums of f' (e.g.
//     n_e = 4 diag - 2 f'_0 + axis - 3 dJ), the cancellation between m'_e
//     and -2 rho' happening exactly inside the sum;
//   * quadratic differences a b / rho - a0 b0 / rho0 are
//     N / rho0^2 * (1 - rho'/rho) with N = rho0 (a0 b' + a' b0 + a' b')
//     - rho' a0 b0: rho = rho0 + rho' is rounded only inside the small
//     correction rho'/rho.
// Measured against the FP64 oracle this keeps the 2000-step plane wave of
// the optimized sets within ~5e-7 of the amplitude (3.5e-6 with the
// straightforward FP32 formulation).
//
// PRECISE: carry the rates and reference-state constants as hi + lo pairs
// (FP32 storage); the 16-bit storage types round far more than the lo parts
// correct and use the hi parts alone.
// SCALED: f holds f' * scale (FP16 storage) and stays in those units: the
// step is linear in f' except for the three quadratic terms and rho'/rho,
// which take the factor inv_scale; with power-of-two scales this equals
// collide-then-rescale bit for bit and saves the per-population rescaling.
template <bool PRECISE, bool SCALED>
__device__ __forceinline__ void collide_dev(float &f0, float &f1, float &f2, float &f3,
                                            float &f4, float &f5, float &f6, float &f7,
                                            float &f8, const DevParams &P) {
  const float s13 = f1 + f3, s24 = f2 + f4;
  const float d13 = f1 - f3, d24 = f2 - f4;
  const float s57 = f5 + f7, s68 = f6 + f8;
  const float d57 = f5 - f7, d68 = f6 - f8;
  const float axis = s13 + s24;
  const float diag = s57 + s68;
  const float dxd = d57 - d68;  // f5 - f6 - f7 + f8
  const float dyd = d57 + d68;  // f5 + f6 - f7 - f8
  const float rho_p = f0 + axis + diag;
  const float jx_p = d13 + dxd;
  const float jy_p = d24 + dyd;

  // m^eq(rho, j) - m^eq(rho0, j0) for the three quadratic terms
  const float rho_phys = SCALED ? rho_p * P.inv_scale : rho_p;
  // rho'/rho by the hardware reciprocal (within 2 ulp): c only scales the
  // O(amplitude^2) quadratic terms below, and unlike an IEEE division it has
  // no slow path for non-finite operands, so a lattice that has gone
  // unstable costs no more per node than a healthy one
  const float c = rho_phys * rcp_approx(P.rho0 + rho_phys);
  const float jxx = SCALED ? (jx_p * jx_p) * P.inv_scale : jx_p * jx_p;
  const float jyy = SCALED ? (jy_p * jy_p) * P.inv_scale : jy_p * jy_p;
  const float jxy = SCALED ? (jx_p * jy_p) * P.inv_scale : jx_p * jy_p;
  const float tx = fmaf(2.0f * P.jx0, jx_p, jxx);  // jx^2 - jx0^2
  const float ty = fmaf(2.0f * P.jy0, jy_p, jyy);
  const float txy = fmaf(P.jx0, jy_p, fmaf(jx_p, P.jy0, jxy));  // jx jy - jx0 jy0
  const float nj =
      mul_hl<PRECISE>(fmaf(P.rho0, tx + ty, -mul_hl<PRECISE>(rho_p, P.q0h, P.q0l)), P.i2h, P.i2l);
  const float np =
      mul_hl<PRECISE>(fmaf(P.rho0, tx - ty, -mul_hl<PRECISE>(rho_p, P.d0h, P.d0l)), P.i2h, P.i2l);
  const float nx =
      mul_hl<PRECISE>(fmaf(P.rho0, txy, -mul_hl<PRECISE>(rho_p, P.x0h, P.x0l)), P.i2h, P.i2l);
  const float djsq = fmaf(-nj, c, nj);  // |j|^2/rho - |j0|^2/rho0
  const float dpxx = fmaf(-np, c, np);  // (jx^2 - jy^2)/rho - (..)0/rho0
  const float dpxy = fmaf(-nx, c, nx);  // jx jy / rho - jx0 jy0 / rho0

  // non-equilibrium parts, each straight from partial sums
  const float n3 = fmaf(-3.0f, djsq, fmaf(4.0f, diag, fmaf(-2.0f, f0, axis)));  // e' + 2 rho' - 3 dJ
  const float n4 = fmaf(3.0f, djsq, 3.0f * (f0 - axis));             // eps' - rho' + 3 dJ
  const float n5 = fmaf(2.0f, dxd, -d13);                            // qx' + jx'
  const float n6 = fmaf(2.0f, dyd, -d24);                            // qy' + jy'
  const float n7 = (s13 - s24) - dpxx;
  const float n8 = (s57 - s68) - dpxy;
  const float r3 = mul_hl<PRECISE>(n3, P.k3, P.l3);
  const float r4 = mul_hl<PRECISE>(n4, P.k4, P.l4);
  const float r5 = mul_hl<PRECISE>(n5, P.k5, P.l5);
  const float r6 = mul_hl<PRECISE>(n6, P.k6, P.l6);
  const float r7 = mul_hl<PRECISE>(n7, P.k7, P.l7);
  const float r8 = mul_hl<PRECISE>(n8, P.k8, P.l8);

  // f <- f - M^T r: columns of M for each velocity
  const float a = fmaf(2.0f, r4, r3);     // axis velocities: -r3 - 2 r4
  const float b = fmaf(2.0f, r3, r4);     // diagonals: 2 r3 + r4
  f0 -= 4.0f * (r4 - r3);
  f1 += fmaf(2.0f, r5, a - r7);
  f3 += fmaf(-2.0f, r5, a - r7);
  f2 += fmaf(2.0f, r6, a + r7);
  f4 += fmaf(-2.0f, r6, a + r7);
  f5 -= b + r5 + r6 + r8;
  f6 -= b - r5 + r6 - r8;
  f7 -= b - r5 - r6 + r8;
  f8 -= b + r5 - r6 - r8;
}

// ------------------------------------------------------------------
// Two nodes at once with the packed FP32 instructions of sm_100 and later
// (add / sub / mul / fma .rn.f32x2): each does the work of two scalar
// instructions, lane by lane with the scalar instruction's IEEE rounding.
// The 16-bit storage types unpack two nodes per 32-bit word, so the pair is
// already there; at 36 B per node their step is bound by instruction issue
// more than by HBM, and this halves the collision's issue slots (measured on
// one 8192^2 lattice: BF16 6.69 -> 6.99 TB/s, FP16 6.82 -> 6.86 TB/s).
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F2 f2s(float a) { return f2(a, a); }
__device__ __forceinline__ void f2split(F2 a, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// a * b + c, one rounding per lane
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// The per-lattice constants collide_pair multiplies by, each broadcast to
// both lanes of an F2; negations and doublings are folded in (exact in
// FP32, so every source of them gives the same bits).
enum PairConst {
  PC_IS, PC_R0, PC_2JX, PC_2JY, PC_JX, PC_JY, PC_I2, PC_NQ0, PC_ND0, PC_NX0,
  PC_K3, PC_K4, PC_NK5, PC_NK6, PC_K7, PC_K8, PC_COUNT
};

__host__ __device__ __forceinline__ float pair_const(const DevParams &P, int c) {
  switch (c) {
    case PC_IS: return P.inv_scale;
    case PC_R0: return P.rho0;
    case PC_2JX: return 2.0f * P.jx0;
    case PC_2JY: return 2.0f * P.jy0;
    case PC_JX: return P.jx0;
    case PC_JY: return P.jy0;
    case PC_I2: return P.i2h;
    case PC_NQ0: return -P.q0h;
    case PC_ND0: return -P.d0h;
    case PC_NX0: return -P.x0h;
    case PC_K3: return P.k3;
    case PC_K4: return P.k4;
    case PC_NK5: return -P.k5;
    case PC_NK6: return -P.k6;
    case PC_K7: return P.k7;
    default: return P.k8;
  }
}

// two constants (collide_pair takes them k, k + 1 with k even: a source in
// shared memory reads both with one 16-byte load)
struct F2x2 {
  F2 a, b;
};

// The constants straight from a DevParams (kernel parameters of a single
// lattice, or an entry in global memory)
struct ParamPairs {
  static constexpr bool kTable = false;
  const DevParams &P;
  __device__ __forceinline__ F2x2 two(PairConst c) const {
    return {f2s(pair_const(P, c)), f2s(pair_const(P, c + 1))};
  }
};

// collide_dev<false, SCALED> for two nodes, one per lane of the F2 values:
// the same formulation (partial sums, quadratic differences through
// rho'/rho, hi parts of the constants), written with explicit multiply-adds.
// Negations are folded into constants or operands where that is exact
// (a sign flip never rounds), so no extra instruction carries them.
template <bool SCALED, typename K>
__device__ __forceinline__ void collide_pair(F2 &f0, F2 &f1, F2 &f2_, F2 &f3, F2 &f4, F2 &f5,
                                             F2 &f6, F2 &f7, F2 &f8, const K &P) {
  const F2 s13 = f1 + f3, s24 = f2_ + f4;
  const F2 d13 = f1 - f3, d24 = f2_ - f4;
  const F2 s57 = f5 + f7, s68 = f6 + f8;
  const F2 d57 = f5 - f7, d68 = f6 - f8;
  const F2 axis = s13 + s24;
  const F2 diag = s57 + s68;
  const F2 dxd = d57 - d68;
  const F2 dyd = d57 + d68;
  const F2 rho_p = (f0 + axis) + diag;
  const F2 jx_p = d13 + dxd;
  const F2 jy_p = d24 + dyd;

  const F2x2 c0 = P.two(PC_IS), c2j = P.two(PC_2JX), cj = P.two(PC_JX);
  const F2 IS = c0.a, R0 = c0.b;
  const F2 rho_phys = SCALED ? rho_p * IS : rho_p;
  // -rho'/rho per lane by the hardware reciprocal (the sign folded into
  // the numerator, which is exact): rho' * rcp(rho) without __fdividef's
  // handling of denominators above 2^126, the same bits below.  FP16 with
  // its constants in constant memory keeps __fdividef: the bare reciprocal
  // spills 80 instead of 64 bytes there at the 72-register cap (BF16 64
  // instead of 100): 39.8 against 39.3 us per step on five lattices of 6.7 M
  // nodes, 5.35 against 5.18 on three of 0.5 M
  const F2 den = R0 + rho_phys;
  float rl, rh, dl, dh;
  f2split(rho_phys, rl, rh);
  f2split(den, dl, dh);
  F2 nc;
  if constexpr (SCALED && K::kTable) nc = f2(__fdividef(-rl, dl), __fdividef(-rh, dh));
  else nc = f2(-rl * rcp_approx(dl), -rh * rcp_approx(dh));
  F2 jxx = jx_p * jx_p, jyy = jy_p * jy_p, jxy = jx_p * jy_p;
  if (SCALED) {
    jxx = jxx * IS;
    jyy = jyy * IS;
    jxy = jxy * IS;
  }
  const F2 tx = fma2(c2j.a, jx_p, jxx);  // jx^2 - jx0^2
  const F2 ty = fma2(c2j.b, jy_p, jyy);
  const F2 txy = fma2(cj.a, jy_p, fma2(jx_p, cj.b, jxy));
  const F2x2 ci = P.two(PC_I2), cn = P.two(PC_ND0);
  const F2 I2 = ci.a;
  const F2 nj = fma2(R0, tx + ty, rho_p * ci.b) * I2;
  const F2 np = fma2(R0, tx - ty, rho_p * cn.a) * I2;
  const F2 nx = fma2(R0, txy, rho_p * cn.b) * I2;
  const F2 djsq = fma2(nj, nc, nj);  // |j|^2/rho - |j0|^2/rho0
  const F2 dpxx = fma2(np, nc, np);
  const F2 dpxy = fma2(nx, nc, nx);

  const F2 n3 = fma2(f2s(-3.0f), djsq, fma2(f2s(4.0f), diag, fma2(f2s(-2.0f), f0, axis)));
  const F2 n4 = fma2(f2s(3.0f), djsq, f2s(3.0f) * (f0 - axis));
  // m5 = -(qx' + jx'), m6 = -(qy' + jy'): their rates enter negated
  const F2 m5 = fma2(f2s(-2.0f), dxd, d13);
  const F2 m6 = fma2(f2s(-2.0f), dyd, d24);
  const F2 n7 = (s13 - s24) - dpxx;
  const F2 n8 = (s57 - s68) - dpxy;
  const F2x2 k34 = P.two(PC_K3), k56 = P.two(PC_NK5), k78 = P.two(PC_K7);
  const F2 r3 = n3 * k34.a;
  const F2 r4 = n4 * k34.b;
  const F2 r5 = m5 * k56.a;
  const F2 r6 = m6 * k56.b;
  const F2 r7 = n7 * k78.a;
  const F2 r8 = n8 * k78.b;

  const F2 TWO = f2s(2.0f), NTWO = f2s(-2.0f);
  const F2 a = fma2(TWO, r4, r3);  // axis velocities: -r3 - 2 r4
  const F2 b = fma2(TWO, r3, r4);  // diagonals: 2 r3 + r4
  f0 = fma2(f2s(-4.0f), r4 - r3, f0);
  const F2 ax = a - r7, ay = a + r7;
  f1 = f1 + fma2(TWO, r5, ax);
  f3 = f3 + fma2(NTWO, r5, ax);
  f2_ = f2_ + fma2(TWO, r6, ay);
  f4 = f4 + fma2(NTWO, r6, ay);
  const F2 bp = b + r5, bm = b - r5;
  f5 = f5 - ((bp + r6) + r8);
  f6 = f6 - ((bm + r6) - r8);
  f7 = f7 - ((bm - r6) + r8);
  f8 = f8 - ((bp - r6) - r8);
}

// The FP32 constants of collide_pair_hl: the high parts with their low parts
// (collide_dev's PRECISE form), each broadcast to both lanes of a pair,
// doublings and negations folded in (exact).
enum HlConst {
  HL_R0, HL_2JX, HL_2JY, HL_JX, HL_JY, HL_PAD,       // rho0, 2 j0, j0
  HL_NQ0H, HL_NQ0L, HL_ND0H, HL_ND0L, HL_NX0H, HL_NX0L,  // -|j0|^2, ...
  HL_I2H, HL_I2L,                                    // 1 / rho0^2
  HL_K3H, HL_K3L, HL_K4H, HL_K4L, HL_NK5H, HL_NK5L,  // rates / D
  HL_NK6H, HL_NK6L, HL_K7H, HL_K7L, HL_K8H, HL_K8L,
  HL_COUNT
};

__host__ __device__ __forceinline__ float hl_const(const DevParams &P, int c) {
  switch (c) {
    case HL_R0: return P.rho0;
    case HL_2JX: return 2.0f * P.jx0;
    case HL_2JY: return 2.0f * P.jy0;
    case HL_JX: return P.jx0;
    case HL_JY:
    case HL_PAD: return P.jy0;
    case HL_NQ0H: return -P.q0h;
    case HL_NQ0L: return -P.q0l;
    case HL_ND0H: return -P.d0h;
    case HL_ND0L: return -P.d0l;
    case HL_NX0H: return -P.x0h;
    case HL_NX0L: return -P.x0l;
    case HL_I2H: return P.i2h;
    case HL_I2L: return P.i2l;
    case HL_K3H: return P.k3;
    case HL_K3L: return P.l3;
    case HL_K4H: return P.k4;
    case HL_K4L: return P.l4;
    case HL_NK5H: return -P.k5;
    case HL_NK5L: return -P.l5;
    case HL_NK6H: return -P.k6;
    case HL_NK6L: return -P.l6;
    case HL_K7H: return P.k7;
    case HL_K7L: return P.l7;
    case HL_K8H: return P.k8;
    default: return P.l8;
  }
}

// the broadcast pairs, as a kernel parameter or in shared memory; two(k), k
// even, reads constants k and k + 1 with one 16-byte load
struct alignas(16) HlPairs {
  float2 c[HL_COUNT];
  __device__ __forceinline__ F2x2 two(HlConst k) const {
    const float4 v = *reinterpret_cast<const float4 *>(c + k);
    return {f2(v.x, v.y), f2(v.z, v.w)};
  }
};

inline HlPairs hl_pairs(const DevParams &P) {
  HlPairs H;
  for (int k = 0; k < HL_COUNT; ++k) H.c[k].x = H.c[k].y = hl_const(P, k);
  return H;
}

// a * (h + l), as mul_hl<true>
__device__ __forceinline__ F2 mul_hl2(F2 a, const F2x2 &k) { return fma2(a, k.a, a * k.b); }

// collide_dev<true, false> (FP32 storage) for two nodes, one per lane: the
// same operations in the same order, multiply-adds written out in both, so
// each lane's result equals the scalar form's bit for bit however the compiler
// contracts the rest (products by powers of two, exact either way).
template <typename K>
__device__ __forceinline__ void collide_pair_hl(F2 &f0, F2 &f1, F2 &f2_, F2 &f3, F2 &f4, F2 &f5,
                                                F2 &f6, F2 &f7, F2 &f8, const K &P) {
  const F2 s13 = f1 + f3, s24 = f2_ + f4;
  const F2 d13 = f1 - f3, d24 = f2_ - f4;
  const F2 s57 = f5 + f7, s68 = f6 + f8;
  const F2 d57 = f5 - f7, d68 = f6 - f8;
  const F2 axis = s13 + s24;
  const F2 diag = s57 + s68;
  const F2 dxd = d57 - d68;
  const F2 dyd = d57 + d68;
  const F2 rho_p = (f0 + axis) + diag;
  const F2 jx_p = d13 + dxd;
  const F2 jy_p = d24 + dyd;

  // -rho'/rho per lane (the sign folded into the numerator, exact)
  const F2x2 c0 = P.two(HL_R0), c1 = P.two(HL_2JY);  // rho0, 2 jx0; 2 jy0, jx0
  const F2 R0 = c0.a;
  const F2 den = R0 + rho_p;
  float rl, rh, dl, dh;
  f2split(rho_p, rl, rh);
  f2split(den, dl, dh);
  const F2 nc = f2(-rl * rcp_approx(dl), -rh * rcp_approx(dh));
  const F2 tx = fma2(c0.b, jx_p, jx_p * jx_p);
  const F2 ty = fma2(c1.a, jy_p, jy_p * jy_p);
  const F2 txy = fma2(c1.b, jy_p, fma2(jx_p, P.two(HL_JY).a, jx_p * jy_p));
  const F2x2 i2 = P.two(HL_I2H);
  const F2 nj = mul_hl2(fma2(R0, tx + ty, mul_hl2(rho_p, P.two(HL_NQ0H))), i2);
  const F2 np = mul_hl2(fma2(R0, tx - ty, mul_hl2(rho_p, P.two(HL_ND0H))), i2);
  const F2 nx = mul_hl2(fma2(R0, txy, mul_hl2(rho_p, P.two(HL_NX0H))), i2);
  const F2 djsq = fma2(nj, nc, nj);
  const F2 dpxx = fma2(np, nc, np);
  const F2 dpxy = fma2(nx, nc, nx);

  const F2 TWO = f2s(2.0f), NTWO = f2s(-2.0f);
  const F2 n3 = fma2(f2s(-3.0f), djsq, fma2(f2s(4.0f), diag, fma2(NTWO, f0, axis)));
  const F2 n4 = fma2(f2s(3.0f), djsq, f2s(3.0f) * (f0 - axis));
  const F2 m5 = fma2(NTWO, dxd, d13);  // -n5, -n6: their rates come negated
  const F2 m6 = fma2(NTWO, dyd, d24);
  const F2 n7 = (s13 - s24) - dpxx;
  const F2 n8 = (s57 - s68) - dpxy;
  const F2 r3 = mul_hl2(n3, P.two(HL_K3H));
  const F2 r4 = mul_hl2(n4, P.two(HL_K4H));
  const F2 r5 = mul_hl2(m5, P.two(HL_NK5H));
  const F2 r6 = mul_hl2(m6, P.two(HL_NK6H));
  const F2 r7 = mul_hl2(n7, P.two(HL_K7H));
  const F2 r8 = mul_hl2(n8, P.two(HL_K8H));

  const F2 a = fma2(TWO, r4, r3);
  const F2 b = fma2(TWO, r3, r4);
  f0 = fma2(f2s(-4.0f), r4 - r3, f0);
  const F2 ax = a - r7, ay = a + r7;
  f1 = f1 + fma2(TWO, r5, ax);
  f3 = f3 + fma2(NTWO, r5, ax);
  f2_ = f2_ + fma2(TWO, r6, ay);
  f4 = f4 + fma2(NTWO, r6, ay);
  const F2 bp = b + r5, bm = b - r5;
  f5 = f5 - ((bp + r6) + r8);
  f6 = f6 - ((bm + r6) - r8);
  f7 = f7 - ((bm - r6) + r8);
  f8 = f8 - ((bp - r6) - r8);
}

// ------------------------------------------------------------------
// FP64 deviation storage (LBM_F64DEV): the deviation form of collide_dev in
// FP64 with fused multiply-adds -- fewer and cheaper FP64 operations than the
// plain path's canonical operation order, and rounding at the size of the
// perturbation, not of f.  GB300's FP64 pipe (two operations per clock and
// SM) bounds the step, so the operations are counted: 71 per node where the
// FP32 form's order takes 89.  With rho0 / rho in place of 1 - rho'/rho, the
// quadratic differences are (N - rho' j0 j0 / rho0) / rho, two of them folded
// into the sums they are subtracted from, and each relaxation rate rides in a
// multiply-add where its moment is used once with either sign.  2048^2: 731
// -> 592 us per step (7.1 GLUPS), with the same error against 64 bits.
struct DevParams64 {
  double rho0, jx0, jy0, jx2, jy2;  // reference state, 2 jx0, 2 jy0
  double k3, k4, k5, k6, k7, k8;    // s_e/36, 3 s_eps/36, s_qx/12, s_qy/12, s_pxx/4, s_pxy/4
  double k6x2;                      // 2 s_qy/12
  double q0, d0, x0;                // -|j0|^2, -(jx0^2 - jy0^2), -jx0 jy0, over rho0
};

__device__ __forceinline__ void collide_dev64(double &f0, double &f1, double &f2, double &f3,
                                              double &f4, double &f5, double &f6, double &f7,
                                              double &f8, const DevParams64 &P) {
  const double s13 = f1 + f3, s24 = f2 + f4;
  const double d13 = f1 - f3, d24 = f2 - f4;
  const double s57 = f5 + f7, s68 = f6 + f8;
  const double d57 = f5 - f7, d68 = f6 - f8;
  const double axis = s13 + s24;
  const double diag = s57 + s68;
  const double dxd = d57 - d68;
  const double dyd = d57 + d68;
  const double rho_p = f0 + axis + diag;
  const double jx_p = d13 + dxd;
  const double jy_p = d24 + dyd;
  // 1/rho by the hardware's approximate FP64 reciprocal r (relative error e
  // of about 2^-20) and r (1 + e + e^2), which leaves e^3
  const double den = P.rho0 + rho_p;
  double rinv;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(rinv) : "d"(den));
  const double e = fma(-den, rinv, 1.0);
  rinv = fma(rinv, fma(e, e, e), rinv);
  const double jxx = jx_p * (jx_p + P.jx2);  // jx^2 - jx0^2
  const double jyt = jy_p + P.jy2;           // (jy^2 - jy0^2) / j'y
  const double txy = fma(jx_p, jy_p + P.jy0, P.jx0 * jy_p);  // jx jy - jx0 jy0
  const double nj = fma(rho_p, P.q0, fma(jy_p, jyt, jxx));
  const double np = fma(rho_p, P.d0, fma(-jy_p, jyt, jxx));
  const double nx = fma(rho_p, P.x0, txy);
  const double djsq = nj * rinv;  // |j|^2/rho - |j0|^2/rho0
  const double n3 = fma(-3.0, djsq, fma(4.0, diag, fma(-2.0, f0, axis)));
  const double n4 = djsq + (f0 - axis);  // a third of eps' - rho' + 3 dJ
  const double n5 = fma(2.0, dxd, -d13);
  const double n6 = fma(2.0, dyd, -d24);
  const double n7 = fma(-np, rinv, s13 - s24);
  const double n8 = fma(-nx, rinv, s57 - s68);
  const double r3 = n3 * P.k3, r4 = n4 * P.k4, r5 = n5 * P.k5;
  const double a = fma(2.0, r4, r3);
  const double b = fma(2.0, r3, r4);
  const double ax = fma(-n7, P.k7, a), ay = fma(n7, P.k7, a);
  const double bp = fma(n8, P.k8, b), bm = fma(-n8, P.k8, b);
  const double rp = fma(n6, P.k6, r5), rm = fma(-n6, P.k6, r5);
  f0 = fma(-4.0, r4 - r3, f0);
  f1 += fma(2.0, r5, ax);
  f3 += fma(-2.0, r5, ax);
  f2 += fma(n6, P.k6x2, ay);
  f4 += fma(-n6, P.k6x2, ay);
  f5 -= bp + rp;
  f6 -= bm - rm;
  f7 -= bp - rp;
  f8 -= bm + rm;
}

// FP64 rates of the plain path: s3 = s_e, s4 = s_eps, s5 = s_qx, s6 = s_qy,
// s7 = s_pxx, s8 = s_pxy.
struct F64Params {
  double s3, s4, s5, s6, s7, s8;
};

// 1 / b correctly rounded (Markstein, IBM J. Res. Dev. 34 (1990) 111): r (1 +
// e + e^2), e = 1 - b r exact, takes the hardware's approximation (a relative
// error of about 2^-20) to within 2^-60 before its rounding, so to the nearest
// FP64 number or, next to a midpoint, the other one; one more step r + r (1 -
// b r), its difference exact, then rounds correctly for every significand but
// the one of all ones.  recip_rounds says that b is not that one and, like its
// reciprocal, far from overflow and underflow.
__device__ __forceinline__ bool recip_rounds(double b) {  // 2^-500 <= |b| < 2^500
  const unsigned hi = (unsigned)__double2hiint(b), lo = (unsigned)__double2loint(b);
  return ((hi >> 20) & 0x7ffu) - 523u < 1000u && ((hi | 0xfff00000u) & lo) != 0xffffffffu;
}
__device__ __forceinline__ double recip(double b) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  const double e = fma(-b, r, 1.0);
  r = fma(r, fma(e, e, e), r);
  return fma(r, fma(-b, r, 1.0), r);
}

// a / b correctly rounded, for the three quotients of one collision by the
// same b: with y = 1 / b correctly rounded (recip), q = a y and the exact
// remainder r = a - b q give the correctly rounded quotient q + r y
// (Markstein).  With y one unit off, as two Newton-Raphson steps from the
// hardware's approximation may leave it, a / b next to a midpoint rounds
// wrongly: 2^-8 / (1 - 2^-53) did.  The argument needs b, the a's and the
// quotients far from overflow and underflow; `fast` says so from the
// exponents (a zero a is fine), and anything else takes the ordinary
// division.  Three quotients cost 5 + 3 x 3 FP64 operations instead of three
// times the compiler's division sequence.
struct Quotients {
  double b, y;
  bool fast;
  static __device__ __forceinline__ bool normal(double v) {  // 2^-500 <= |v| < 2^500
    const unsigned e = ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
    return e - 523u < 1000u;
  }
  __device__ __forceinline__ Quotients(double b_, double a0, double a1, double a2) : b(b_) {
    auto ok = [](double a) { return normal(a) || a_zero(a); };
    fast = recip_rounds(b) && ok(a0) && ok(a1) && ok(a2);
    y = recip(b);
  }
  static __device__ __forceinline__ bool a_zero(double a) {
    return (((unsigned)__double2hiint(a) << 1) | (unsigned)__double2loint(a)) == 0u;
  }
  __device__ __forceinline__ double operator()(double a) const {
    const double q = a * y;
    return fma(fma(-b, q, a), y, q);
  }
};

// Plain FP64 collision of the full populations, with the results of a plain
// matrix-vector implementation of section 2.1 (each moment the sum over j =
// 0..8 of M_kj f_j taken left to right; m^eq as written in section 2.3
// ((-2 rho) + (3 |j|^2)/rho, ...); r_k = s_k (m_k - m^eq_k); f_i - sum over k
// = 0..8 of (M_ki / D_k) r_k left to right; zero terms skipped), bit for
// bit.  GB300's FP64 pipe bounds the step, so operations that cannot change
// a bit are saved: products by powers of two are exact, so they ride in
// fused multiply-adds and are shared between rows that scale alike ((2 a) +
// (2 b) rounds to 2 (a + b)); the three divisions share one reciprocal
// (Quotients).  119 instead of ~185 FP64 instructions per node.  Compile
// without multiply-add contraction (-fmad=false).
__device__ __forceinline__ void collide_f64(double (&f)[9], const F64Params &P) {
  const double rho = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
  const double d13 = f[1] - f[3], d24 = f[2] - f[4];
  const double jx = d13 + f[5] - f[6] - f[7] + f[8];
  const double jy = d24 + f[5] + f[6] - f[7] - f[8];
  const double e = fma(2.0, f[8], fma(2.0, f[7], fma(2.0, f[6], fma(2.0, f[5],
                       fma(-4.0, f[0], -f[1]) - f[2] - f[3] - f[4]))));
  const double eps = fma(2.0, fma(2.0, f[0], -f[1]) - f[2] - f[3] - f[4], f[5]) + f[6] + f[7] +
                     f[8];
  const double qx = fma(-2.0, d13, f[5]) - f[6] - f[7] + f[8];
  const double qy = fma(-2.0, d24, f[5]) + f[6] - f[7] - f[8];
  const double pxx = f[1] - f[2] + f[3] - f[4];
  const double pxy = f[5] - f[6] + f[7] - f[8];

  const double jxx = jx * jx, jyy = jy * jy;
  const double a0 = 3.0 * (jxx + jyy), a1 = jxx - jyy, a2 = jx * jy;
  const Quotients Q(rho, a0, a1, a2);
  double dj = Q(a0), pxx_eq = Q(a1), pxy_eq = Q(a2);
  if (!Q.fast) {
    dj = a0 / rho;
    pxx_eq = a1 / rho;
    pxy_eq = a2 / rho;
  }
  const double e_eq = fma(-2.0, rho, dj);
  const double eps_eq = rho - dj;

  constexpr double c36 = 1.0 / 36.0, c12 = 1.0 / 12.0;
  const double p3 = c36 * (P.s3 * (e - e_eq));
  const double p4 = c36 * (P.s4 * (eps - eps_eq));
  const double p5 = c12 * (P.s5 * (qx + jx));
  const double p6 = c12 * (P.s6 * (qy + jy));
  const double r7 = P.s7 * (pxx - pxx_eq);
  const double r8 = P.s8 * (pxy - pxy_eq);

  const double t = fma(-2.0, p4, -p3), u = fma(2.0, p3, p4);
  f[0] = fma(-4.0, p4 - p3, f[0]);
  f[1] = f[1] - fma(0.25, r7, fma(-2.0, p5, t));
  f[2] = f[2] - fma(-0.25, r7, fma(-2.0, p6, t));
  f[3] = f[3] - fma(0.25, r7, fma(2.0, p5, t));
  f[4] = f[4] - fma(-0.25, r7, fma(2.0, p6, t));
  const double up = u + p5, um = u - p5;
  f[5] = f[5] - fma(0.25, r8, up + p6);
  f[6] = f[6] - fma(-0.25, r8, um + p6);
  f[7] = f[7] - fma(0.25, r8, um - p6);
  f[8] = f[8] - fma(-0.25, r8, up - p6);
}

}  // namespace lbm
