// Device functions of one WSBM node-pair block (eq. weakly_bm; block form A_ij of Sec. III),
// shared by the entry generator and the matrix-free product.
#pragma once
#include "hankel.cuh"
#include "wsbm_internal.h"

#define WSBM_4PI 12.566370614359172954

// Geometric quantities of a pair with the operation order fixed (no contraction): r and the
// arguments z = k r are reproducible bit for bit by any IEEE double implementation.
struct PairGeom {
  double r, ir, z0, z1, dnx, dny, nn, c, rs0, rs1;
};

__device__ __forceinline__ void pair_geom(double xi, double yi, double nxi, double nyi, double xj,
                                          double yj, double nxj, double nyj, const Phys& ph,
                                          PairGeom& G) {
  double dx = __dsub_rn(xi, xj);
  double dy = __dsub_rn(yi, yj);
  double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  double r = __dsqrt_rn(r2);
  G.r = r;
  G.z0 = __dmul_rn(ph.k0, r);
  G.z1 = __dmul_rn(ph.k1, r);
  G.dny = __dadd_rn(__dmul_rn(dx, nxj), __dmul_rn(dy, nyj));
  G.dnx = __dadd_rn(__dmul_rn(dx, nxi), __dmul_rn(dy, nyi));
  G.nn = __dadd_rn(__dmul_rn(nxi, nxj), __dmul_rn(nyi, nyj));
  // one reciprocal square root serves both wavenumbers and 1/r
  G.rs0 = rsqrt(G.z0);
  G.rs1 = G.rs0 * ph.s01;
  G.ir = ph.k0 * (G.rs0 * G.rs0);
  G.c = G.dnx * G.dny * (G.ir * G.ir);
}

// Off-diagonal 2x2 block, weight w_j folded in (kernels: G_k = (i/4) H0(kr);
// D: (ik/4) H1 (d.n_y)/r;  D*: -(ik/4) H1 (d.n_x)/r;
// N_k0 - N_k1 = (i/4)[(k0^2 H0(z0) - k1^2 H0(z1)) c + (k0^2 F1(z0) - k1^2 F1(z1))(n_x.n_y - 2c)]).
__device__ __forceinline__ void block_offdiag(const HkTables& T, const Phys& ph, const PairGeom& G,
                                              double wj, double2 e[2][2]) {
  Hk a, b;
  hankel_fp64_rs<true>(T, G.z0, G.rs0, a);
  hankel_fp64_rs<true>(T, G.z1, G.rs1, b);
  const double k0 = ph.k0, k1 = ph.k1;
  double s11 = 0.25 * wj * k1 * G.dny * G.ir;  // A11 = i s11 H1(z1)
  e[0][0] = make_double2(-s11 * b.h1i, s11 * b.h1r);
  double s12 = -0.25 * ph.eps1 * wj;  // A12 = i s12 H0(z1)
  e[0][1] = make_double2(-s12 * b.h0i, s12 * b.h0r);
  double q0 = k0 * k0, q1 = k1 * k1;
  double m2c = G.nn - 2.0 * G.c;
  double gr = (q0 * a.h0r - q1 * b.h0r) * G.c + (q0 * a.f1r - q1 * b.f1r) * m2c;
  double gi = (q0 * a.h0i - q1 * b.h0i) * G.c + (q0 * a.f1i - q1 * b.f1i) * m2c;
  double inv4k0 = 0.25 * ph.inv_k0;
  double t1 = 0.25 * k0 * G.dny * G.ir;
  // A21 = w [ i t1 H1(z0) + alpha dN ],  alpha dN = -(1/(4 k0)) (gr + i gi)
  e[1][0] = make_double2(wj * (-t1 * a.h1i - inv4k0 * gr), wj * (t1 * a.h1r - inv4k0 * gi));
  // A22 = w [ -i (eps0/4) H0(z0) - (d.n_x/(4 k0 r)) (eps0 k0 H1(z0) - eps1 k1 H1(z1)) ]
  double u = G.dnx * G.ir * inv4k0;
  double vr = ph.eps0 * k0 * a.h1r - ph.eps1 * k1 * b.h1r;
  double vi = ph.eps0 * k0 * a.h1i - ph.eps1 * k1 * b.h1i;
  e[1][1] = make_double2(wj * (0.25 * ph.eps0 * a.h0i - u * vr),
                         wj * (-0.25 * ph.eps0 * a.h0r - u * vi));
}

// r^2 of a pair in the fixed operation order (no contraction).
__device__ __forceinline__ double pair_r2(double dx, double dy) {
  return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}
__device__ __forceinline__ bool pair_is_fixed(const Phys& ph, double r2) {
  const int h = __double2hiint(r2);
  return h > ph.fix_lo && h < ph.fix_hi;
}

// 1/sqrt(x) to an ulp for normal x: the hardware's seed y (rsqrt.approx.ftz.f64, about 22 bits) and one
// step of third order.  With e = 1 - x y^2, 1/sqrt(x) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + O(e^3)),
// the binomial series; the next term, 5 e^3/16, is below 2^-60.
__device__ __forceinline__ double rsqrt3(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// The same for any x > 0 (subnormal and infinite ones through the library function).
__device__ __forceinline__ double rsqrt3_any(double x) {
  const int h = __double2hiint(x);
  return h >= 0x00100000 && h < 0x7FF00000 ? rsqrt3(x) : rsqrt(x);
}

// sqrt(x) from y = 1/sqrt(x) by one Newton step: r = x y, then r + (x - r^2) y / 2, the residual from a
// fused multiply-add.  Correctly rounded wherever compared with sqrt().
__device__ __forceinline__ double sqrt_from(double x, double y) {
  const double r = x * y;
  return fma(fma(-r, r, x), __hiloint2double(__double2hiint(y) - 0x100000, __double2loint(y)), r);
}

// Off-diagonal block of a pair with both arguments in the range of hankel_fixed.  Same formulas
// as block_offdiag, with three savings on the FP64 pipe, which bounds every pair kernel (one
// FP64 instruction costs as much issue time as 64 others): the Hankel values come from the
// integer pipe; r (correctly rounded) and 1/r share one reciprocal
// square root; and the amplitudes sqrt(2/(pi k r)) and every constant are folded into eight real
// factors of the unit-amplitude values, so that an entry is two to five multiply-adds.  The
// 1/(k r)^2 poles of F1 cancel in N_k0 - N_k1 and are left out (at z >= 1.5 they are no larger than
// the values they stand beside).
// 71 FP64 instructions where the general path takes about 185.
__device__ __forceinline__ void block_fixed(const HkTables& T, const Phys& ph, double dx, double dy, double r2, double nxi, double nyi,
                                          double nxj, double nyj, double wj, double2 e[2][2]) {
  const double ir = rsqrt3(r2);
  const double r = sqrt_from(r2, ir);
  const double z0 = __dmul_rn(ph.k0, r), z1 = __dmul_rn(ph.k1, r);
  HxUnit a, b;
  hankel_fixed(T.near_, z0, ir * ph.inv_k0, a);
  hankel_fixed(T.near_, z1, ir * ph.inv_k1, b);
  const double dny = __dadd_rn(__dmul_rn(dx, nxj), __dmul_rn(dy, nyj)) * ir;
  const double dnx = __dadd_rn(__dmul_rn(dx, nxi), __dmul_rn(dy, nyi)) * ir;
  const double nn = __dadd_rn(__dmul_rn(nxi, nxj), __dmul_rn(nyi, nyj));
  const double c = dnx * dny, m2c = fma(-2.0, c, nn);
  const double w0 = wj * rsqrt3(z0);
  const double v0 = w0 * ph.c_v, t0 = v0 * dny, c0 = v0 * c;  // t1 H1(z0), k0 H0(z0) c
  const double mr = w0 * m2c * ir, d0 = mr * ph.c_d0, d1 = mr * ph.c_d1;
  const double c1 = w0 * c * ph.c_c1;
  const double s11 = w0 * dny * ph.c_s11, s12 = w0 * ph.c_s12;
  const double e0 = w0 * ph.c_e0, u0 = e0 * dnx, u1 = w0 * dnx * ph.c_u1;
  e[0][0] = make_double2(-s11 * b.i1, s11 * b.r1);
  e[0][1] = make_double2(-s12 * b.i0, s12 * b.r0);
  e[1][0] = make_double2(fma(-t0, a.i1, fma(-c0, a.r0, fma(-d0, a.r1, fma(c1, b.r0, d1 * b.r1)))),
                         fma(t0, a.r1, fma(-c0, a.i0, fma(-d0, a.i1, fma(c1, b.i0, d1 * b.i1)))));
  e[1][1] = make_double2(fma(e0, a.i0, fma(-u0, a.r1, u1 * b.r1)), fma(-e0, a.r0, fma(-u0, a.i1, u1 * b.i1)));
}

// Off-diagonal block of target (xi, yi, nxi, nyi) and source (xj, yj, nxj, nyj, wj).
__device__ __forceinline__ void pair_block(const HkTables& T, const Phys& ph, double xi, double yi, double nxi,
                                           double nyi, double xj, double yj, double nxj, double nyj, double wj,
                                           double2 e[2][2]) {
  const double dx = __dsub_rn(xi, xj), dy = __dsub_rn(yi, yj), r2 = pair_r2(dx, dy);
  if (pair_is_fixed(ph, r2)) {
    block_fixed(T, ph, dx, dy, r2, nxi, nyi, nxj, nyj, wj, e);
  } else {
    PairGeom G;
    pair_geom(xi, yi, nxi, nyi, xj, yj, nxj, nyj, ph, G);
    block_offdiag(T, ph, G, wj, e);
  }
}

// Diagonal 2x2 block: one-point corrected trapezoidal rule.  A kernel a ln|x-y| + b gets the
// weight w_i [a ln(w_i/2pi) + b(x_i, x_i)]; D and D* tend to -kappa/(4 pi).
__device__ __forceinline__ void block_diag(const Phys& ph, double wi, double kap, double2 e[2][2]) {
  const double k0 = ph.k0, k1 = ph.k1;
  double L0 = log(k0 * wi / WSBM_4PI);
  double L1 = log(k1 * wi / WSBM_4PI);
  double S0r = -wi * (WSBM_EULER + L0) / (2.0 * WSBM_PI), Si = 0.25 * wi;
  double S1r = -wi * (WSBM_EULER + L1) / (2.0 * WSBM_PI);
  double Dd = -wi * kap / WSBM_4PI;
  double f0 = k0 * k0 * (L0 + WSBM_EULER - 0.5);
  double f1 = k1 * k1 * (L1 + WSBM_EULER - 0.5);
  double dNr = -wi * (f0 - f1) / WSBM_4PI;
  double dNi = wi * (k0 * k0 - k1 * k1) / 8.0;
  e[0][0] = make_double2(Dd + 0.5, 0.0);
  e[0][1] = make_double2(-ph.eps1 * S1r, -ph.eps1 * Si);
  e[1][0] = make_double2(Dd - 0.5 - dNi / k0, dNr / k0);
  e[1][1] = make_double2(-ph.eps0 * S0r,
                         -ph.eps0 * Si - ((ph.eps0 - ph.eps1) * Dd + 0.5 * (ph.eps0 + ph.eps1)) / k0);
}
