// Small triangular solves of the dense kernels, one warp per column.
#pragma once
#include "cplx.cuh"

// x <- T^-1 x for the leading nb x nb triangle at T (nb <= 32 NS): unit lower, or (UPPER) upper
// with its diagonal, a zero diagonal entry giving a zero.  The column sits in the lanes'
// registers (row 32 s + lane in x[s]).  Columns of T come through shared memory 32 at a time
// (`stage`: 32 x 32 NS values, shared by the CTA's warps), so a step is a broadcast of x_t and a
// few multiply-adds off shared memory: a chain of about 100 clocks a row instead of a chain of
// global loads (a 128 x 128 inverse takes 88 us spread over 128 SMs; 1.7 ms with a thread per
// column).  An upper triangle's columns are scaled by the reciprocals of its diagonal as they are
// staged, so no step multiplies by them.  Every thread of the CTA has to call it with the same T and
// nb; warps that are not `active` only help with the staging.  `first` (the same for every thread):
// the slot where the nonzeros of every column of the CTA begin (end, if UPPER); the slots before it are
// skipped, and of the warp's column the steps before its row `own`, whose x_t are zero.  Both matter
// where many matrices fill the FP64 pipe: 4096 pairs of 64 x 64 inverses 27.7 ms without, 14.0 ms with.
template <int NS, bool UPPER>
__device__ __forceinline__ void tri_solve_warp(const double2* __restrict__ T, int64_t ldt, int nb, double2 (&x)[NS],
                                               double2* stage, double2* dinv, bool active = true,
                                               int first = UPPER ? NS - 1 : 0, int own = UPPER ? 32 * NS - 1 : 0) {
  constexpr int LD = 32 * NS;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    const int s = UPPER ? NS - 1 - q : q;
    const int t0 = s * 32;
    if (t0 >= nb || (UPPER ? s > first : s < first)) continue;  // the same for every thread of the CTA
    const int te = min(32, nb - t0);
    const int i0 = UPPER ? 0 : t0, i1 = UPPER ? t0 + te : nb;
    __syncthreads();
    for (int e = threadIdx.x; e < te * LD; e += blockDim.x) {
      const int tt = e / LD, i = e - tt * LD;
      if (i >= i0 && i < i1) stage[e] = T[i + (int64_t)(t0 + tt) * ldt];
    }
    __syncthreads();
    if (UPPER) {
      if (threadIdx.x < te) {
        const double2 v = stage[threadIdx.x * LD + t0 + threadIdx.x];
        dinv[threadIdx.x] =
            v.x == 0.0 && v.y == 0.0 ? make_double2(0.0, 0.0) : cdiv(make_double2(1.0, 0.0), v);
      }
      __syncthreads();
      for (int e = threadIdx.x; e < te * LD; e += blockDim.x) {
        const int tt = e / LD, i = e - tt * LD;
        if (i < t0 + tt) stage[e] = cmul(stage[e], dinv[tt]);
      }
      __syncthreads();
    }
    if (!active) continue;
    for (int k = max(0, UPPER ? t0 + te - 1 - own : own - t0); k < te; ++k) {
      const int tt = UPPER ? te - 1 - k : k;
      const double2* col = stage + tt * LD;
      double2 xt;
      xt.x = __shfl_sync(0xFFFFFFFFu, x[s].x, tt);
      xt.y = __shfl_sync(0xFFFFFFFFu, x[s].y, tt);
#pragma unroll
      for (int r = 0; r < NS; ++r) {
        const int i = r * 32 + lane;
        if (UPPER ? (r < s || (r == s && lane < tt)) : (r > s || (r == s && lane > tt)))
          if (UPPER || i < nb) x[r] = cfms(col[i], xt, x[r]);
      }
    }
    if (UPPER && lane < te) x[s] = cmul(x[s], dinv[lane]);
  }
}

// Column j of the inverse of that triangle into out[0 .. nb); first: as above.
template <int NS, bool UPPER>
__device__ __forceinline__ void tri_inverse_column(const double2* __restrict__ T, int64_t ldt, int nb, int j,
                                                   double2* __restrict__ out, double2* stage, double2* dinv,
                                                   bool active, int first) {
  const int lane = threadIdx.x & 31;
  double2 x[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) x[s] = make_double2(s * 32 + lane == j ? 1.0 : 0.0, 0.0);
  tri_solve_warp<NS, UPPER>(T, ldt, nb, x, stage, dinv, active, first, j);
#pragma unroll
  for (int s = 0; s < NS; ++s)
    if (active && j < nb && s * 32 + lane < nb) out[s * 32 + lane] = x[s];
}
