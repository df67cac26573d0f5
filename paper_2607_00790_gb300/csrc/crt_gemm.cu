// Complex128 GEMM of large matrices on the tensor cores from residues (tcgen05 + TMA + TMEM).
//
//   C (m x n) = beta C + alpha A (m x k) B (k x n),   complex128, column-major.
//
// Same scaling as tc_gemm.cu: row i of A and column j of B become integers X = x 2^(56 - e) with
// |Re X|, |Im X| < 2^55.  Instead of products of 8-bit digits (34 digit pairs x 4 real products per
// complex one) the integer product is formed modulo 14 pairwise coprime numbers (the integer modular
// form of the Ozaki scheme) and put together by the Chinese remainder theorem:
//
//  1. Moduli.  Every prime factor of a modulus p is 1 modulo 4, so -1 has a square root iota mod p
//     and a complex product splits into two real ones: with A+- = Re A +- iota Im A (likewise B),
//     P+- = sum A+- B+- = Re C +- iota Im C (mod p).  28 real products in all (136 for the digits).
//     p <= 509: the balanced residues are at most 254 in size, exact in BF16, and 256 products of
//     them sum to less than 2^24, exact in FP32.
//  2. Range.  The product of the moduli is M > 2^122; |Re C|, |Im C| <= 2 k 2^110 < M / 2 for
//     k <= 1024 (longer products run in pieces).
//  3. Reconstruction without large integers.  C / M = frac(sum_p r_p w_p) with fixed fractions w_p:
//     the sum is kept modulo 1 in a wrapping 64-bit integer plus an FP32 sum of the parts of the w_p
//     below 2^-64 (about 2^-75 of M, 2^-60 of a typical entry), so every modulus costs a few FP32 and
//     integer operations per entry and nothing is stored per modulus.  C / M becomes a double by
//     integer operations.  Where all the inputs of an entry are multiples of a power of two (integers,
//     say) that makes its exact value representable, the result is rounded to that multiple, so
//     products of small integers are exact.
//
// Error: the rounding of X to 56 bits, as in tc_gemm.cu; nothing is dropped.
//
// Kernel: one CTA per SM, persistent over 128 x 48 complex tiles.  Warp 0 issues the TMA loads (a
// 5-stage ring of 32-deep K blocks of four planes, 64-byte swizzled rows), warp 1 the MMAs (128 x 48 x
// 16, the four accumulators in turn) into two TMEM buffers (P+ and P- of two moduli each); warps 4-11
// reduce them: two threads per row, 24 columns each, 6 registers of running sums per entry (setmaxnreg
// moves the registers over; 64 columns a CTA spill).  Bound by the instructions of that reduction (about
// 25 issue slots per entry and modulus, 160 to make the double), 6 clocks per entry and SM: 2.44 ms at
// 8192 x 8192 x 256.  Every CTA loads whole A tiles: pairs of CTAs that shared them were no faster (2.5
// ms), since the loads are not the bound, and each had to outlive the other's arrivals.
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "dense.h"
#include "tc_ptx.cuh"

#define CR_NP 14             // moduli
#define CR_PL (2 * CR_NP)    // planes per operand
#define CR_BM 128            // rows per tile
#define CR_BN 48             // complex columns per tile
#define CR_TC (CR_BN / 2)    // columns per epilogue thread: 6 CR_TC registers of running sums
#define CR_BK 32             // K values per stage (64-byte rows)
#define CR_G 4               // planes per stage: P+ and P- of two moduli
#define CR_KC 256            // K values per exact accumulation
#define CR_KMAX 1024         // K values per reconstruction
#define CR_STAGES 5
#define CR_A_BYTES (CR_BM * CR_BK * 2)
#define CR_B_BYTES (CR_BN * CR_BK * 2)
#define CR_STAGE (CR_G * (CR_A_BYTES + CR_B_BYTES))
#define CR_SMEM (CR_STAGES * CR_STAGE + 256 + 1024)
#define CR_THREADS 384
#define CR_EPI 256
// registers a thread of the four warps that issue and of the epilogue, out of those of the launch (168 each):
// an increase beyond the launch's total would wait for ever, so crt_registers() checks it
#define CR_REGS_ISSUE 40
#define CR_REGS_EPI 232
#define CR_NBUF 2            // TMEM buffers of CR_G x 64 columns (the accumulators use CR_BN of each 64)
#define CR_FEWBITS 40        // a row or column of values of at most so many significant bits
#define CR_LOW_NONE 1000000  // lowest set bit of an all-zero row or column

struct CrtMod {
  int p, inv, m1, m2, iota;     // 2^32 / p rounded up, 2^19 and 2^38 mod p, square root of -1
  int h, off;                   // (p - 1) / 2, and h + 1024 p
  float fp, ip;                 // p, 1 / p
  uint32_t wl, wh, vl, vh;      // fractions (unit 2^-64) of r+ + r- in Re C / M and of r+ - r- in Im C / M
  float wx, vx;                 // their parts below 2^-64
};
struct CrtTable {
  CrtMod mod[CR_NP];
  uint64_t base_r, base_i;  // what the float-to-integer offset of one accumulation adds to the sums
  uint64_t mn;              // M = mn 2^(mbits - 64), mn >= 2^63
  int mbits, pad;
};

// One product (or strip of one).
struct CrtArgs {
  CrtTable t;
  double2* C;
  int64_t ldc;
  const int2 *rexp, *cexp;  // {scale exponent, lowest set bit} of each row of A and column of B
  double2 alpha, beta;
  int m, n, kb;             // kb: K blocks of CR_BK
  int mode;                 // 0: C = A B, 1: C -= A B, 2: general
  int tiles_m, tiles_n;     // 128 x 48 tiles
  int group;                // row tiles per raster group
};

// K-major tile of 64-byte rows, 64-byte swizzle (atoms of 8 rows, 512 bytes apart).
__device__ __forceinline__ uint64_t cr_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
         (uint64_t)4 << 61;
}
__device__ __forceinline__ void cr_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accum) {
  // BF16 x BF16 -> FP32, both K-major, M = 128, N = CR_BN
  constexpr uint32_t idesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(CR_BN >> 3) << 17) | ((uint32_t)(CR_BM >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accum));
}

// ------------------------------------------------------------------ residues ----
__device__ __forceinline__ int low_bit(double v) {  // exponent of the lowest set bit
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FF);
  const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (E ? 1ull << 52 : 0);
  return mant ? (E ? E : 1) - 1075 + __ffsll((long long)mant) - 1 : CR_LOW_NONE;
}
// X = v 2^(56 - e), rounded half up in magnitude when v has bits below (|v| < 2^(e-1), |X| < 2^55).
__device__ __forceinline__ int64_t fix56(double v, int e) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FF);
  const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (E ? 1ull << 52 : 0);
  const int sh = (E > 0 ? E : 1) - 1075 + 56 - e;
  int64_t X;
  if (mant == 0 || sh <= -64)
    X = 0;
  else if (sh >= 0)
    X = (int64_t)(mant << sh);
  else
    X = (int64_t)((mant + (1ull << (-sh - 1))) >> (-sh));
  return b >> 63 ? -X : X;
}
struct Limbs {
  int x0, x1, x2;
};
__device__ __forceinline__ Limbs limbs(int64_t X) {
  return Limbs{(int)(X & 0x7FFFF), (int)((X >> 19) & 0x7FFFF), (int)(X >> 38)};
}
// X modulo p up to a multiple of p: in (-p / 8, 9 p / 8).
__device__ __forceinline__ int residue(const Limbs& x, const CrtMod& c) {
  const int t = x.x2 * c.m2 + x.x1 * c.m1 + x.x0;  // below 2^29
  return t - __mulhi(t, c.inv) * c.p;
}
// Balanced residue of |t| < 1024 p as an exact float (the quotient of the nonnegative t + 1024 p +
// (p - 1) / 2 is exact: its error is below 2^-12 of a unit).
__device__ __forceinline__ float balanced(int t, const CrtMod& c) {
  const int w = t + c.off, r = w - __mulhi(w, c.inv) * c.p - c.h;
  return __int_as_float(0x4B400000 + r) - 12582912.0f;
}
__device__ __forceinline__ void split_mod(const Limbs& re, const Limbs& im, const CrtMod& c, float& plus, float& minus) {
  const int r = residue(re, c), i = residue(im, c) * c.iota;
  plus = balanced(r + i, c);
  minus = balanced(r - i, c);
}

// {scale exponent, lowest set bit} of the rows of A (m x k): 32 rows a CTA, 32 warps over the columns.
__global__ void __launch_bounds__(1024) k_crt_row_exp(const double2* __restrict__ A, int64_t lda, int m, int k,
                                                      int2* __restrict__ out) {
  __shared__ uint64_t red[32][33];
  __shared__ int redl[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  uint64_t mx = 0;
  int lo = CR_LOW_NONE;
  if (i < m) {
#pragma unroll 4
    for (int l = warp; l < k; l += 32) {
      const double2 v = A[i + (int64_t)l * lda];
      mx = max(mx, max(abs_bits(v.x), abs_bits(v.y)));
      lo = min(lo, min(low_bit(v.x), low_bit(v.y)));
    }
  }
  red[warp][lane] = mx;
  redl[warp][lane] = lo;
  __syncthreads();
  mx = red[lane][warp];
  lo = redl[lane][warp];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)mx, o);
    mx = max(mx, (uint64_t)other);
    lo = min(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
  }
  const int r = blockIdx.x * 32 + warp;
  if (lane == 0 && r < m) out[r] = make_int2(scale_exp(mx), lo);
}

// The same for the columns of B (k x n): one warp per column.
__global__ void __launch_bounds__(256) k_crt_col_exp(const double2* __restrict__ B, int64_t ldb, int k, int n,
                                                     int2* __restrict__ out) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= n) return;
  uint64_t mx = 0;
  int lo = CR_LOW_NONE;
#pragma unroll 4
  for (int l = lane; l < k; l += 32) {
    const double2 v = B[l + (int64_t)j * ldb];
    mx = max(mx, max(abs_bits(v.x), abs_bits(v.y)));
    lo = min(lo, min(low_bit(v.x), low_bit(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)mx, o);
    mx = max(mx, (uint64_t)other);
    lo = min(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
  }
  if (lane == 0) out[j] = make_int2(scale_exp(mx), lo);
}

// Residue planes of A (m x k), [CR_PL][m][Kp] with zeros beyond k: 32 rows x 32 columns a CTA, staged
// through shared memory (reads along a column, writes along a row), 7 moduli at a time.
__global__ void __launch_bounds__(256) k_crt_split_a(const __grid_constant__ CrtTable t, const double2* __restrict__ A,
                                                     int64_t lda, int m, int k, int Kp, const int2* __restrict__ exps,
                                                     __nv_bfloat16* __restrict__ P) {
  __shared__ __nv_bfloat16 s[CR_NP][32][34];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i0 = blockIdx.x * 32, l0 = blockIdx.y * 32, i = i0 + tx;
  Limbs re[4], im[4];
  const int e = i < m ? exps[i].x : 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int l = l0 + ty + 8 * q;
    const double2 v = i < m && l < k ? A[i + (int64_t)l * lda] : make_double2(0.0, 0.0);
    re[q] = limbs(fix56(v.x, e));
    im[q] = limbs(fix56(v.y, e));
  }
  const int64_t plane = (int64_t)m * Kp;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (half) __syncthreads();
#pragma unroll
    for (int jj = 0; jj < CR_NP / 2; ++jj) {
      const CrtMod& c = t.mod[half * (CR_NP / 2) + jj];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float p, mi;
        split_mod(re[q], im[q], c, p, mi);
        s[2 * jj][tx][ty + 8 * q] = __float2bfloat16_rn(p);
        s[2 * jj + 1][tx][ty + 8 * q] = __float2bfloat16_rn(mi);
      }
    }
    __syncthreads();
    for (int w = threadIdx.x; w < CR_NP * 32 * 16; w += 256) {
      const int pl = w / (32 * 16), r = (w / 16) % 32, c2 = w % 16;
      if (i0 + r >= m) continue;
      __nv_bfloat162 v;
      v.x = s[pl][r][2 * c2];
      v.y = s[pl][r][2 * c2 + 1];
      *reinterpret_cast<__nv_bfloat162*>(P + (half * CR_NP + pl) * plane + (int64_t)(i0 + r) * Kp + l0 + 2 * c2) = v;
    }
  }
}

// Residue planes of B (k x n), [CR_PL][n][Kp]: a thread per two rows of a column.
__global__ void __launch_bounds__(128) k_crt_split_b(const __grid_constant__ CrtTable t, const double2* __restrict__ B,
                                                     int64_t ldb, int k, int n, int Kp, const int2* __restrict__ exps,
                                                     __nv_bfloat16* __restrict__ P) {
  const int64_t w = blockIdx.x * (int64_t)128 + threadIdx.x;
  const int half = Kp / 2;
  const int64_t j = w / half;
  if (j >= n) return;
  const int l = 2 * (int)(w - j * half), e = exps[j].x;
  Limbs re[2], im[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double2 v = l + q < k ? B[l + q + j * ldb] : make_double2(0.0, 0.0);
    re[q] = limbs(fix56(v.x, e));
    im[q] = limbs(fix56(v.y, e));
  }
  const int64_t plane = (int64_t)n * Kp;
#pragma unroll
  for (int jj = 0; jj < CR_NP; ++jj) {
    float p[2], mi[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) split_mod(re[q], im[q], t.mod[jj], p[q], mi[q]);
    __nv_bfloat16* o = P + (int64_t)(2 * jj) * plane + j * Kp + l;
    *reinterpret_cast<__nv_bfloat162*>(o) = __floats2bfloat162_rn(p[0], p[1]);
    *reinterpret_cast<__nv_bfloat162*>(o + plane) = __floats2bfloat162_rn(mi[0], mi[1]);
  }
}

// ------------------------------------------------------------------ the product ----
// a - p rint(a / p), exact for integers |a| <= 2^24.
__device__ __forceinline__ float reduce_mod(float a, const CrtMod& c) {
  const float q = fmaf(a, c.ip, 12582912.0f) - 12582912.0f;
  return fmaf(-c.fp, q, a);
}

// f + x w modulo 2^64.
__device__ __forceinline__ uint64_t mad_frac(uint32_t x, uint32_t wl, uint32_t wh, uint64_t f) {
  uint64_t r;
  asm("{\n\t.reg .u32 lo, hi;\n\t.reg .u64 t;\n\t"
      "mad.wide.u32 t, %1, %2, %4;\n\t"
      "mov.b64 {lo, hi}, t;\n\t"
      "mad.lo.u32 hi, %1, %3, hi;\n\t"
      "mov.b64 %0, {lo, hi};\n\t}"
      : "=l"(r)
      : "r"(x), "r"(wl), "r"(wh), "l"(f));
  return r;
}

// (acc + low) 2^-64 M 2^ex as a double (acc: signed), rounded once; low is below 2^22 in size.  E:
// its biased exponent, which the double carries modulo 2^11 (crt_fix handles the rare E outside the
// normal range).
__device__ __forceinline__ double crt_double(uint64_t acc, float low, const CrtTable& t, int ex, int& E) {
  int64_t a = (int64_t)acc;
  // 8 bits below the unit where there is room
  const int sh = a < (1ll << 54) && a > -(1ll << 54) ? 8 : 0;
  a = (a << sh) + __float2int_rn(low * (sh ? 256.0f : 1.0f));
  const uint64_t s = (uint64_t)(a >> 63), mag = ((uint64_t)a ^ s) - s;
  const int lz = __clzll((long long)mag);  // 64 for zero
  uint64_t h = __umul64hi(mag << (lz & 63), t.mn);  // at least 2^62
  const int z = (int)(h >> 63) ^ 1;
  h <<= z;
  const uint64_t mant = (h >> 11) + ((h >> 10) & 1);  // 53 bits (a carry moves into the exponent)
  E = mag ? 1022 + t.mbits - lz - z - sh + ex : 1;
  return __longlong_as_double((long long)(((mag ? (uint64_t)(E - 1) << 52 : 0) + mant) | (s << 63)));
}
// x (biased exponent E modulo 2^11) brought into range and, where few significant bits make the exact
// value a multiple of 2^quant that a double can tell from its neighbours, rounded to one.
__device__ __forceinline__ double crt_fix(double x, int E, int quant) {
  const long long b = __double_as_longlong(x);
  if ((unsigned)(E - 1) > 2043u)  // the mantissa with the exponent of 1, scaled in one rounding
    x = ldexp(__longlong_as_double((b & 0x800FFFFFFFFFFFFFll) | (1023ll << 52)), E - 1023);
  if (E - 1023 < 51 + quant && quant > -900 && quant < 900) {
    const double r = __hiloint2double(((quant + 52 + 1023) << 20) | 0x80000, 0);  // 1.5 2^52 2^quant
    x = __dsub_rn(__dadd_rn(x, r), r);
  }
  return x;
}

// The finished sums of one tile into C: row i, columns j0 .. j0 + CR_TC - 1.  Four columns at a time, their
// loads in flight together; the sums move down four places after each (a few MOVs), so that this is a
// loop: unrolled, its code ran at the speed of instruction fetches.
template <bool SLOW>
__device__ __forceinline__ void crt_finish(const CrtArgs& a, uint64_t (&fr)[CR_TC], uint64_t (&fi)[CR_TC], float (&lr)[CR_TC],
                                           float (&li)[CR_TC], int2 er, int2 ecl, int i, int j0) {
  double2* cp = a.C + i + (int64_t)j0 * a.ldc;
  const bool in = i < a.m, old = in && (a.mode == 1 || (a.mode == 2 && (a.beta.x != 0.0 || a.beta.y != 0.0)));
  const int nc = in ? min(CR_TC, a.n - j0) : 0;
#pragma unroll 1
  for (int c0 = 0; c0 < CR_TC; c0 += 4) {
    double2 o[4], r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      o[q] = old && c0 + q < nc ? cp[(int64_t)(c0 + q) * a.ldc] : make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int ex = er.x + __shfl_sync(0xFFFFFFFFu, ecl.x, c0 + q) - 112;
      int Er, Ei;
      r[q].x = crt_double(fr[q], lr[q], a.t, ex, Er);
      r[q].y = crt_double(fi[q], li[q], a.t, ex, Ei);
      if (SLOW) {
        const int quant = er.y + __shfl_sync(0xFFFFFFFFu, ecl.y, c0 + q);
        r[q].x = crt_fix(r[q].x, Er, quant);
        r[q].y = crt_fix(r[q].y, Ei, quant);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (a.mode == 1) {
        r[q] = make_double2(o[q].x - r[q].x, o[q].y - r[q].y);
      } else if (a.mode == 2) {
        const double2 x = r[q];
        r[q] = make_double2(a.alpha.x * x.x - a.alpha.y * x.y, a.alpha.x * x.y + a.alpha.y * x.x);
        if (old) {
          r[q].x += a.beta.x * o[q].x - a.beta.y * o[q].y;
          r[q].y += a.beta.x * o[q].y + a.beta.y * o[q].x;
        }
      }
      if (c0 + q < nc) cp[(int64_t)(c0 + q) * a.ldc] = r[q];
    }
#pragma unroll
    for (int c = 0; c < CR_TC - 4; ++c) {
      fr[c] = fr[c + 4];
      fi[c] = fi[c + 4];
      lr[c] = lr[c + 4];
      li[c] = li[c + 4];
    }
  }
}

__global__ void __launch_bounds__(CR_THREADS, 1)
    k_zgemm_crt(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CrtArgs a) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = smem_raw + (base - raw);
  const uint32_t bars = base + CR_STAGES * CR_STAGE;
  const uint32_t full0 = bars, empty0 = bars + 8 * CR_STAGES, tfull0 = bars + 16 * CR_STAGES,
                 tempty0 = tfull0 + 8 * CR_NBUF;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + CR_STAGES * CR_STAGE + 16 * CR_STAGES + 16 * CR_NBUF);
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int ntiles = a.tiles_m * a.tiles_n;
  const int nchunks = (a.kb + CR_KC / CR_BK - 1) / (CR_KC / CR_BK);

  if (threadIdx.x == 0) {
    for (int s = 0; s < CR_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < CR_NBUF; ++s) {
      mbar_init(tfull0 + 8 * s, 1);
      mbar_init(tempty0 + 8 * s, CR_EPI);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // tile t -> (row tile, column tile): groups of a.group row tiles, so that the CTAs running at the
  // same time share operands in L2
  auto coords = [&](int t, int& tm, int& tn) {
    const int per = a.group * a.tiles_n, g = t / per, q = t % per, gm = min(a.group, a.tiles_m - g * a.group);
    tm = g * a.group + q % gm;
    tn = q / gm;
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(CR_REGS_ISSUE));
    if (warp == 0 && lane == 0) {
      // -------------------------------------------------------------- TMA producer
      uint32_t it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int tm, tn;
        coords(t, tm, tn);
        for (int kc = 0; kc < a.kb && ok; kc += CR_KC / CR_BK) {
          const int ke = min(a.kb, kc + CR_KC / CR_BK);
          for (int g = 0; g < CR_PL / CR_G && ok; ++g)
            for (int kb = kc; kb < ke; ++kb, ++it) {
              const uint32_t s = it % CR_STAGES, ph = (it / CR_STAGES) & 1;
              if (!(ok = mbar_wait(empty0 + 8 * s, ph ^ 1))) break;
              const uint32_t full = full0 + 8 * s, sa = base + s * CR_STAGE, sb = sa + CR_G * CR_A_BYTES;
              mbar_expect_tx(full, CR_STAGE);
#pragma unroll
              for (int q = 0; q < CR_G; ++q) {
                tma_load_3d(sa + q * CR_A_BYTES, &mapA, full, kb * CR_BK, tm * CR_BM, g * CR_G + q);
                tma_load_3d(sb + q * CR_B_BYTES, &mapB, full, kb * CR_BK, tn * CR_BN, g * CR_G + q);
              }
            }
        }
      }
      // every load into this CTA has landed (bounded) before it leaves
      for (uint32_t s = 0; s < CR_STAGES; ++s) {
        if (it <= s) continue;
        const uint32_t last = s + ((it - 1 - s) / CR_STAGES) * CR_STAGES;
        mbar_wait(full0 + 8 * s, (last / CR_STAGES) & 1);
      }
    } else if (warp == 1 && lane == 0) {
      // -------------------------------------------------------------- MMA issuer
      uint32_t it = 0, u = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        for (int kc = 0; kc < a.kb && ok; kc += CR_KC / CR_BK) {
          const int ke = min(a.kb, kc + CR_KC / CR_BK);
          for (int g = 0; g < CR_PL / CR_G && ok; ++g, ++u) {
            const uint32_t b = u % CR_NBUF;
            if (!(ok = mbar_wait(tempty0 + 8 * b, ((u / CR_NBUF) & 1) ^ 1))) break;
            tc_fence_after();
            for (int kb = kc; kb < ke; ++kb, ++it) {
              const uint32_t s = it % CR_STAGES, ph = (it / CR_STAGES) & 1;
              if (!(ok = mbar_wait(full0 + 8 * s, ph))) break;
              tc_fence_after();
              const uint32_t sa = base + s * CR_STAGE, sb = sa + CR_G * CR_A_BYTES;
#pragma unroll
              for (int kk = 0; kk < CR_BK / 16; ++kk)  // 16 values = 32 bytes = 2 units of the address
#pragma unroll
                for (int q = 0; q < CR_G; ++q)  // four accumulators in turn: no product waits for the last
                  cr_mma(tmem + (b * CR_G + q) * 64, cr_desc(sa + q * CR_A_BYTES) + 2 * kk,
                         cr_desc(sb + q * CR_B_BYTES) + 2 * kk, kb > kc || kk > 0 ? 1u : 0u);
              tc_commit(empty0 + 8 * s);
            }
            if (ok) tc_commit(tfull0 + 8 * b);
          }
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 4-11)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(CR_REGS_EPI));
    const int quad = warp & 3, half = (warp - 4) >> 2;  // TMEM lanes, and which half of the columns
    const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + half * CR_TC;
    uint32_t u = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      int tm, tn;
      coords(t, tm, tn);
      uint64_t fr[CR_TC], fi[CR_TC];
      float lr[CR_TC], li[CR_TC];
#pragma unroll
      for (int c = 0; c < CR_TC; ++c) {
        fr[c] = 0 - a.t.base_r * (uint64_t)nchunks;
        fi[c] = 0 - a.t.base_i * (uint64_t)nchunks;
        lr[c] = li[c] = 0.0f;
      }
      for (int e = 0; e < nchunks * (CR_NP / 2); ++e, ++u) {
        const uint32_t b = u % CR_NBUF;
        if (!(ok = mbar_wait(tfull0 + 8 * b, (u / CR_NBUF) & 1))) break;
        tc_fence_after();
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const CrtMod& c = a.t.mod[2 * (e % (CR_NP / 2)) + h];
          const uint32_t tb = tq + (b * CR_G + 2 * h) * 64;
#pragma unroll
          for (int g = 0; g < CR_TC / 8; ++g) {
            float vp[8], vm[8];
            tmem_ld8(tb + g * 8, vp);
            tmem_ld8(tb + 64 + g * 8, vm);
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 8; ++x) {
              const int y = g * 8 + x;
              const float rp = reduce_mod(vp[x], c), rm = reduce_mod(vm[x], c);
              const float sp = rp + rm, sd = rp - rm;  // integers of at most p in size
              lr[y] = fmaf(sp, c.wx, lr[y]);
              li[y] = fmaf(sd, c.vx, li[y]);
              fr[y] = mad_frac(__float_as_uint(sp + 12582912.0f), c.wl, c.wh, fr[y]);
              fi[y] = mad_frac(__float_as_uint(sd + 12582912.0f), c.vl, c.vh, fi[y]);
            }
          }
        }
        tc_fence_before();
        mbar_arrive(tempty0 + 8 * b);
      }
      if (!ok) break;
      // scales of this thread's row and of column j0 + lane (dealt out by shuffles)
      const int i = tm * CR_BM + quad * 32 + lane, j0 = tn * CR_BN + half * CR_TC;
      const int2 er = i < a.m ? a.rexp[i] : make_int2(0, -1000);
      const int2 ecl = lane < CR_TC && j0 + lane < a.n ? a.cexp[j0 + lane] : make_int2(0, -1000);
      // crt_fix is needed only for extreme scales, or where a row and a column have few significant bits
      const bool slow = __any_sync(0xFFFFFFFFu, abs(er.x) > 400 || abs(ecl.x) > 400) ||
                        (__any_sync(0xFFFFFFFFu, er.y > er.x - CR_FEWBITS) &&
                         __any_sync(0xFFFFFFFFu, ecl.y > ecl.x - CR_FEWBITS));
      if (slow)
        crt_finish<true>(a, fr, fi, lr, li, er, ecl, i, j0);
      else
        crt_finish<false>(a, fr, fi, lr, li, er, ecl, i, j0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// -------------------------------------------------------------------- host side ----
static const CrtTable& crt_table() {
  static const CrtTable t = [] {
    const int ps[CR_NP] = {509, 505, 493, 481, 461, 457, 449, 433, 421, 409, 401, 397, 389, 373};
    CrtTable r;
    memset(&r, 0, sizeof(r));
    unsigned __int128 M = 1;
    for (int p : ps) M *= (unsigned)p;
    auto inverse = [](int v, int p) {  // p is small
      for (int x = 1; x < p; ++x)
        if ((int64_t)v * x % p == 1) return x;
      return 0;
    };
    for (int j = 0; j < CR_NP; ++j) {
      const int p = ps[j];
      CrtMod& c = r.mod[j];
      c.p = p;
      c.inv = (int)(((uint64_t)1 << 32) / (unsigned)p + 1);
      c.m1 = (int)(((uint64_t)1 << 19) % (unsigned)p);
      c.m2 = (int)(((uint64_t)1 << 38) % (unsigned)p);
      for (int x = 1; x < p; ++x)
        if ((int64_t)x * x % p == p - 1) {
          c.iota = x;
          break;
        }
      c.h = (p - 1) / 2;
      c.off = c.h + 1024 * p;
      c.fp = (float)p;
      c.ip = 1.0f / (float)p;
      // sum_p r (M/p) ((M/p)^-1 mod p) / M = sum_p r num / p (mod 1), times 1/2 and 1/(2 iota) mod p
      const int ci = inverse((int)(M / (unsigned)p % (unsigned)p), p);
      const int64_t nr = (int64_t)ci * inverse(2, p) % p, ni = nr * inverse(c.iota, p) % p;
      auto frac = [p](int64_t num, uint32_t& lo, uint32_t& hi, float& x) {
        const unsigned __int128 q = (unsigned __int128)num << 64;
        const uint64_t w = (uint64_t)(q / (unsigned)p);
        lo = (uint32_t)w;
        hi = (uint32_t)(w >> 32);
        x = (float)((double)(uint64_t)(q % (unsigned)p) / p);
        return w;
      };
      r.base_r += (uint64_t)0x4B400000u * frac(nr, c.wl, c.wh, c.wx);
      r.base_i += (uint64_t)0x4B400000u * frac(ni, c.vl, c.vh, c.vx);
    }
    int bits = 0;
    for (unsigned __int128 v = M; v; v >>= 1) ++bits;
    r.mbits = bits;
    r.mn = (uint64_t)(M >> (bits - 64));
    return r;
  }();
  return t;
}

static int crt_map(CUtensorMap* map, void* planes, int64_t rows, int64_t Kp, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return -3;
  cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, (cuuint64_t)CR_PL};
  cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)rows * Kp * 2};
  cuuint32_t box[3] = {CR_BK, (cuuint32_t)box_rows, 1}, es[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, planes, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -3;
}

// The kernel was compiled with the registers that its warps share out.
static bool crt_registers() {
  static const bool ok = [] {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, k_zgemm_crt) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return a.numRegs * CR_THREADS >= (CR_THREADS - CR_EPI) * CR_REGS_ISSUE + CR_EPI * CR_REGS_EPI;
  }();
  return ok;
}

static int64_t crt_kp(int k) { return ((int64_t)std::min(k, CR_KMAX) + CR_BK - 1) / CR_BK * CR_BK; }
static size_t crt_up(size_t b) { return (b + 255) & ~(size_t)255; }
static size_t crt_bytes(int64_t m, int64_t n, int64_t Kp) {
  return crt_up((size_t)CR_PL * m * Kp * 2) + crt_up((size_t)CR_PL * n * Kp * 2) + crt_up((size_t)(m + n) * sizeof(int2));
}

size_t wsbm_zgemm_crt_ws_bytes(int m, int n, int k) { return crt_bytes(m, n, crt_kp(k)); }

// Against the digit planes: large products 8192 x 8192 x 256 2.55 ms against 3.60, x 512 4.50 / 6.34; below k
// = 160 the reduction of the sums, 6 clocks per entry and SM, does not shrink with k (8192 x 8192 x 128 2.04 /
// 2.11).  Smaller results by the waves that their tiles take (128 x 48 here, 128 x 32 there), one of which takes
// up to 1.2 of the other's time with the splits.  Measured for k = 160 to 1000, us at k = 256: 768 x 768 (one
// wave each) 67 / 59, 1024 x 1024 (2, 2) 101 / 87, 1200 x 1200 (2, 3) 105 / 117, 1300 x 1300 (3, 3) 141 / 122,
// 1600 x 1600 (3, 5) 147 / 191, 4000 x 512 (3, 4) 157 / 172, 6000 x 512 (4, 5) 204 / 217.
bool wsbm_zgemm_crt_fits(int m, int n, int k) {
  if (k < 160 || m < 512 || n < 512) return false;
  const int64_t rows = (m + 127) / 128, sms = wsbm_sm_count();
  const int64_t here = (rows * ((n + 47) / 48) + sms - 1) / sms, there = (rows * ((n + 31) / 32) + sms - 1) / sms;
  return 6 * here <= 5 * there;
}

// Do the column-major blocks X (xr x xc) and Y (yr x yc) share an element?  Exact for equal leading
// dimensions (two blocks of one matrix), else by the ranges of their addresses.
static bool blocks_meet(const double2* X, int64_t ldx, int64_t xr, int64_t xc, const double2* Y, int64_t ldy, int64_t yr,
                        int64_t yc) {
  const uintptr_t x0 = (uintptr_t)X, x1 = (uintptr_t)(X + (xc - 1) * ldx + xr);
  const uintptr_t y0 = (uintptr_t)Y, y1 = (uintptr_t)(Y + (yc - 1) * ldy + yr);
  if (x1 <= y0 || y1 <= x0) return false;
  if (ldx != ldy || (y0 - x0) % sizeof(double2)) return true;
  const int64_t d = ((int64_t)y0 - (int64_t)x0) / (int64_t)sizeof(double2);
  const int64_t dr = ((d % ldx) + ldx) % ldx, dc = (d - dr) / ldx;  // Y begins dr rows and dc columns after X
  auto meet = [&](int64_t r, int64_t c) { return r < xr && r + yr > 0 && c < xc && c + yc > 0; };
  return meet(dr, dc) || meet(dr - ldx, dc + 1);
}

// ws_bytes may be less than wsbm_zgemm_crt_ws_bytes: the longer side then goes through in strips
// (-2 if not even a strip of 512 fits, if the registers do not suffice, or if C is written piece by piece while A or B, which it overlaps,
// is still to be read: nothing was launched).
int wsbm_zgemm_crt(int m, int n, int k, double2 alpha, const double2* A, int64_t lda, const double2* B, int64_t ldb,
                   double2 beta, double2* C, int64_t ldc, void* ws, size_t ws_bytes, cudaStream_t st, int group) {
  if (!crt_registers()) return -2;
  const int64_t Kp = crt_kp(k);
  int ms = m, ns = n;
  while (crt_bytes(ms, ns, Kp) > ws_bytes) {
    int& x = ms > ns ? ms : ns;
    if (x <= 512) return -2;
    x = (x / 2 + 127) / 128 * 128;
  }
  if ((k > CR_KMAX || ms < m || ns < n) &&
      (blocks_meet(A, lda, m, k, C, ldc, m, n) || blocks_meet(B, ldb, k, n, C, ldc, m, n)))
    return -2;
  __nv_bfloat16 *PA = (__nv_bfloat16*)ws,
                *PB = (__nv_bfloat16*)((char*)ws + crt_up((size_t)CR_PL * ms * Kp * 2));
  int2* exps = (int2*)((char*)PB + crt_up((size_t)CR_PL * ns * Kp * 2));
  if (wsbm_smem_optin((const void*)k_zgemm_crt, CR_SMEM) != cudaSuccess) return -3;
  CrtArgs a;
  a.t = crt_table();
  a.ldc = ldc;
  a.rexp = exps;
  a.cexp = exps + ms;
  a.group = group;
  for (int k0 = 0; k0 < k; k0 += CR_KMAX) {
    const int kc = std::min(CR_KMAX, k - k0);
    a.alpha = alpha;
    a.beta = k0 ? make_double2(1.0, 0.0) : beta;
    a.kb = (int)((kc + CR_BK - 1) / CR_BK);
    const bool b0 = a.beta.x == 0.0 && a.beta.y == 0.0, b1 = a.beta.x == 1.0 && a.beta.y == 0.0;
    a.mode = alpha.x == 1.0 && alpha.y == 0.0 && b0 ? 0 : alpha.x == -1.0 && alpha.y == 0.0 && b1 ? 1 : 2;
    const int64_t kp = (int64_t)a.kb * CR_BK;
    // A is split once per row strip and B once per pair of strips (one of the two has one strip, unless
    // the work space is very small)
    for (int j0 = 0; j0 < n; j0 += ns) {
      const int nn = std::min(ns, n - j0);
      k_crt_col_exp<<<(nn + 7) / 8, 256, 0, st>>>(B + k0 + (int64_t)j0 * ldb, ldb, kc, nn, exps + ms);
      const int64_t wb = (int64_t)nn * (kp / 2);
      k_crt_split_b<<<(unsigned)((wb + 127) / 128), 128, 0, st>>>(a.t, B + k0 + (int64_t)j0 * ldb, ldb, kc, nn, (int)kp,
                                                                 exps + ms, PB);
      CUtensorMap ma, mb;
      if (crt_map(&mb, PB, nn, kp, CR_BN)) return -3;
      for (int i0 = 0; i0 < m; i0 += ms) {
        const int mm = std::min(ms, m - i0);
        if (j0 == 0 || ms < m) {
          const double2* Ai = A + i0 + (int64_t)k0 * lda;
          k_crt_row_exp<<<(mm + 31) / 32, 1024, 0, st>>>(Ai, lda, mm, kc, exps);
          k_crt_split_a<<<dim3((mm + 31) / 32, (unsigned)(kp / 32)), 256, 0, st>>>(a.t, Ai, lda, mm, kc, (int)kp, exps,
                                                                                  PA);
          wsbm_count_launches(2);
        }
        if (crt_map(&ma, PA, mm, kp, CR_BM)) return -3;
        a.C = C + i0 + (int64_t)j0 * ldc;
        a.m = mm;
        a.n = nn;
        a.tiles_m = (mm + CR_BM - 1) / CR_BM;
        a.tiles_n = (nn + CR_BN - 1) / CR_BN;
        const int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
        const int grid = (int)std::min<int64_t>(tiles, wsbm_sm_count());
        k_zgemm_crt<<<grid, CR_THREADS, CR_SMEM, st>>>(ma, mb, a);
        wsbm_count_launch();
      }
      wsbm_count_launches(2);
    }
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// Error flag of this file's bounded waits: returns -5 and clears it, or 0 (-3 on a CUDA error).
int wsbm_zgemm_crt_status() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)) != cudaSuccess) return -3;
  if (!v) return 0;
  const int zero = 0;
  cudaMemcpyToSymbol(g_tc_error, &zero, sizeof(int));
  return -5;
}
