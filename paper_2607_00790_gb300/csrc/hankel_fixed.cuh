// Hankel functions at 1.5 <= z < 2^20 in 64-bit fixed point on the integer pipe.
//
// GB300 starts 2 FP64 operations per clock and SM against 59 32 x 32 -> 64 bit products and 120
// additions: a 64 x 64 bit product kept to 64 bits (three 32-bit products, two carried additions)
// costs about an eighth of a DFMA.  The phase factor, P_nu, Q_nu and their products are therefore
// formed as 64-bit fractions and only the four results become doubles, by integer operations as
// well.  Each result is within about 2^-58 of the modulus before that rounding, where the FP64
// evaluation loses a few 2^-53.  The matrix-free product of 16384 nodes took 103.8 ms with the FP64
// evaluator (185 FP64 operations a pair, the pipe 90 % busy) and takes 45.5 ms with this one (71 and
// 16 for the product).
//
//   phase   z = m 2^e (53-bit m): m times the 96-bit 2/pi, shifted, gives 2 z / pi modulo 4 to
//           2^-62: the top two bits are the quadrant k of z - pi/4 = (pi/2) (k + x), the rest
//           x + 1/2, so no rounding of the reduction enters
//   E + iF  = i^k (cos(pi x/2) + i sin(pi x/2)), as magnitudes (unit 2^-63) and signs
//   P, Q    from z = 20 on polynomials in 1/z^2, unsigned (1 - P_0 and P_1 - 1 in units of 2^-75,
//           -Q_0 of 2^-70, Q_1 of 2^-69); below it polynomials in 1/z on nine intervals, signed
//
// The functions also compile for the host, where the tests compare them with mpmath.
#pragma once
#include <stdint.h>
#include <string.h>

#include "hankel_fixed.inc"

#ifdef __CUDACC__
#define HX_FN __host__ __device__ __forceinline__
#else
#define HX_FN static inline
#endif

#define HX_Z_LO 1.5             // smallest argument
#define HX_Z_FAR 20.0           // polynomials in 1/z^2 from here on (Z_ASYM of the tables)
#define HX_Z_FAR_WORD 0x40340000
#define HX_Z_HI 1048576.0       // the phase shift needs z < 2^20
#define HX_Z_HI_WORD 0x41300000 // high word of 2^20

// Tables of the intervals below HX_Z_FAR (shared memory on the device).
struct HxNear {
  uint64_t lo[HX_NIV];
  int64_t c[HX_NIV][4][HX_DEG_N + 1];
  int32_t sh[HX_NIV];
};

// H_nu / sqrt(2 / (pi z)), nu = 0, 1.
struct HxUnit {
  double r0, i0, r1, i1;
};

HX_FN uint64_t hx_bits(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return b;
#endif
}
HX_FN double hx_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
HX_FN int hx_clz(uint64_t v) {  // v != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}

// a b / 2^64 without the lowest partial product (below 3 units too small); all, or the upper
// 32 bits, of b.
HX_FN uint64_t hx_mul(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (uint64_t)ah * bh + (((uint64_t)ah * bl) >> 32) + (((uint64_t)al * bh) >> 32);
}
HX_FN uint64_t hx_mul_hi(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32);
  return (uint64_t)ah * bh + (((uint64_t)al * bh) >> 32);
}

// a t / 2^64 for signed a and 0 <= t < 2^63.
HX_FN int64_t hx_mul_s(int64_t a, uint64_t t) {
  const int32_t ah = (int32_t)(a >> 32), th = (int32_t)(t >> 32);
  const uint32_t al = (uint32_t)a, tl = (uint32_t)t;
  return (int64_t)ah * th + (int64_t)(((uint64_t)al * (uint32_t)th) >> 32) + (((int64_t)ah * (int32_t)(tl >> 1)) >> 31);
}

// c_0 - y (c_1 - y (c_2 - ...)), y and the sums as fractions of 2^64.  From coefficient FROM on
// the sums are below 2^-15, so the upper half of y is enough for them.
template <int DEG, int FROM>
HX_FN uint64_t hx_poly(const uint64_t (&c)[DEG + 1], uint64_t y) {
  uint64_t r = c[DEG];
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int j = DEG - 1; j >= 0; --j) r = c[j] - (j + 1 >= FROM ? hx_mul_hi(r, y) : hx_mul(r, y));
  return r;
}

// Signed fixed-point value of unit 2^-62 to double, rounded to nearest.
HX_FN double hx_to_double(int64_t v) {
  const uint64_t s = (uint64_t)(v >> 63), m = ((uint64_t)v ^ s) - s;
  if (m == 0) return 0.0;
  const int lz = hx_clz(m);
  const uint64_t t = m << lz;
  // 53-bit mantissa with its leading one (a carry of the rounding moves into the exponent)
  const uint64_t b = ((uint64_t)(1023 - lz) << 52) + (t >> 11) + ((t >> 10) & 1);
  return hx_double(b | (s << 63));
}

// H_0 and H_1 at HX_Z_LO <= z < HX_Z_HI over the amplitude sqrt(2 / (pi z)); u = 1/z to a few ulp.
HX_FN void hankel_fixed(const HxNear& nt, double z, double u, HxUnit& o) {
  // phase
  uint64_t W;
  {
    const uint32_t c[3] = HX_2_OVER_PI;
    const uint64_t b = hx_bits(z);
    const uint32_t ml = (uint32_t)b, mh = ((uint32_t)(b >> 32) & 0xFFFFFu) | 0x100000u;
    const int sh = 1045 - (int)(b >> 52);  // 3 .. 22
    const uint64_t B = (uint64_t)mh * c[1] + (uint64_t)ml * c[0] + (((uint64_t)ml * c[1]) >> 32) +
                       (((uint64_t)mh * c[2]) >> 32);
    const uint64_t T = (uint64_t)mh * c[0] + (B >> 32);
#ifdef __CUDA_ARCH__
    const uint32_t v0 = (uint32_t)B, v1 = (uint32_t)T, v2 = (uint32_t)(T >> 32);
    W = ((uint64_t)__funnelshift_r(v1, v2, sh) << 32) | __funnelshift_r(v0, v1, sh);
#else
    W = (T << (32 - sh)) | ((uint32_t)B >> sh);
#endif
  }
  const uint32_t k = (uint32_t)(W >> 62);
  const int64_t x = (int64_t)((W << 2) ^ 0x8000000000000000ull);  // fraction - 1/2, unit 2^-64
  const uint64_t xs = (uint64_t)(x >> 63), xm = ((uint64_t)x ^ xs) - xs;
  const uint64_t y = hx_mul(xm, xm);
  const uint64_t cS[HX_DEG_S + 1] = HX_SIN, cC[HX_DEG_C + 1] = HX_COS;
  const uint64_t sn = hx_mul(xm, hx_poly<HX_DEG_S, 5>(cS, y));  // |sin|, unit 2^-63
  const uint64_t cs = hx_poly<HX_DEG_C, 5>(cC, y);              // cos, unit 2^-63
  const uint64_t odd = 0 - (uint64_t)(k & 1);
  const uint64_t aE = cs ^ ((cs ^ sn) & odd), aF = sn ^ ((cs ^ sn) & odd);
  // sign of the sine goes with it; E < 0 for k = 1, 2, F < 0 for k = 2, 3
  const uint64_t sE = (0 - (uint64_t)(((k + 1) >> 1) & 1)) ^ (xs & odd);
  const uint64_t sF = (0 - (uint64_t)(k >> 1)) ^ (xs & ~odd);
  // |E| and |F| times P_nu and -Q_0, Q_1, unit 2^-62
  const uint64_t ub = hx_bits(u), um = ((ub & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
  const int ue = (int)(ub >> 52);
  int64_t e0, f0, e1, f1, qe0, qf0, qe1, qf1;
  const int zhi = (int)(hx_bits(z) >> 32);
  if (zhi >= HX_Z_FAR_WORD) {
    const uint64_t U = um >> (1018 - ue);  // u 2^68
    const uint64_t t = hx_mul(U, U);       // 256 u^2
    const uint64_t cP0[HX_DEG_PQ + 1] = HX_P0, cQ0[HX_DEG_PQ + 1] = HX_Q0, cP1[HX_DEG_PQ + 1] = HX_P1,
                   cQ1[HX_DEG_PQ + 1] = HX_Q1;
    const uint64_t p0 = hx_mul(t, hx_poly<HX_DEG_PQ, 3>(cP0, t)), q0 = hx_mul(U, hx_poly<HX_DEG_PQ, 3>(cQ0, t));
    const uint64_t p1 = hx_mul(t, hx_poly<HX_DEG_PQ, 3>(cP1, t)), q1 = hx_mul(U, hx_poly<HX_DEG_PQ, 3>(cQ1, t));
    e0 = (int64_t)((aE - (hx_mul(aE, p0) >> 11)) >> 1);
    f0 = (int64_t)((aF - (hx_mul(aF, p0) >> 11)) >> 1);
    e1 = (int64_t)((aE >> 1) + (hx_mul(aE, p1) >> 12));
    f1 = (int64_t)((aF >> 1) + (hx_mul(aF, p1) >> 12));
    qe0 = (int64_t)(hx_mul(aE, q0) >> 7);
    qf0 = (int64_t)(hx_mul(aF, q0) >> 7);
    qe1 = (int64_t)(hx_mul(aE, q1) >> 6);
    qf1 = (int64_t)(hx_mul(aF, q1) >> 6);
  } else {
    const int lim[HX_NIV - 1] = HX_IV_HI;
    int iv = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < HX_NIV - 1; ++k) iv += zhi >= lim[k] ? 1 : 0;
    const uint64_t t = ((um >> (1022 - ue)) - nt.lo[iv]) << nt.sh[iv];
    int64_t v[4];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int f = 0; f < 4; ++f) {
      int64_t r = nt.c[iv][f][HX_DEG_N];
#ifdef __CUDACC__
#pragma unroll
#endif
      for (int j = HX_DEG_N - 1; j >= 0; --j) r = nt.c[iv][f][j] + hx_mul_s(r, t);
      v[f] = r;
    }
    const uint64_t hE = aE >> 1, hF = aF >> 1;
    e0 = (int64_t)hE + hx_mul_s(v[0], hE);
    f0 = (int64_t)hF + hx_mul_s(v[0], hF);
    e1 = (int64_t)hE + hx_mul_s(v[2], hE);
    f1 = (int64_t)hF + hx_mul_s(v[2], hF);
    qe0 = -hx_mul_s(v[1], hE);
    qf0 = -hx_mul_s(v[1], hF);
    qe1 = hx_mul_s(v[3], hE);
    qf1 = hx_mul_s(v[3], hF);
  }
  // H_0 = (P E - Q F) + i (P F + Q E),  H_1 = (P F + Q E) + i (Q F - P E)
#define HX_SGN(v, s) (((uint64_t)(v) ^ (s)) - (s))
  o.r0 = hx_to_double((int64_t)(HX_SGN(e0, sE) + HX_SGN(qf0, sF)));
  o.i0 = hx_to_double((int64_t)(HX_SGN(f0, sF) - HX_SGN(qe0, sE)));
  o.r1 = hx_to_double((int64_t)(HX_SGN(f1, sF) + HX_SGN(qe1, sE)));
  o.i1 = hx_to_double((int64_t)(HX_SGN(qf1, sF) - HX_SGN(e1, sE)));
#undef HX_SGN
}
