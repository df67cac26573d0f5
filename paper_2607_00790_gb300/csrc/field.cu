// Field off the curve from the boundary densities by the integral representations (Sec. II:
// once u and q are known on the curve, the solution in each domain follows from them):
//   exterior x:  u_sc(x) = D_k0[u](x) - eps0 S_k0[q](x)      (scattered part)
//   interior x:  u(x)    = eps1 S_k1[q](x) - D_k1[u](x)      (total field)
// S_k[f](x) = sum_j w_j (i/4) H0(k r) f_j,  D_k[f](x) = sum_j w_j (ik/4) H1(k r) (d.n_j)/r f_j,
// d = x - y_j.  The side of x comes from the Laplace double layer of the unit density (Gauss:
// -sum_j w_j (d.n_j)/(2 pi r^2) is 1 inside, 0 outside, up to the quadrature error near the
// curve).  The trapezoidal sums are accurate a few node spacings away from the curve; closer
// targets need a near-singular quadrature, which the paper does not describe.
#include <math.h>

#include <algorithm>

#include "entry_blocks.cuh"
#include "wsbm_internal.h"

namespace {

#define FLD_THREADS 128
// CTAs per SM.  16384 nodes, 3001 targets, 1 and 8 columns: 4.0 and 8.58 ms (16: 3.9 and 8.78; 8: 4.1 and 8.78)
#define FLD_WANT 32

struct FldSlot {
  double x, y, nx, ny, w;
};

// ---- side of the targets.  The Gauss sum is 0 or 1 up to the quadrature error, so FP32 decides
// it nearly everywhere: coordinate differences from (hi, lo) FP32 pairs taken relative to the first
// node (a curve far from the origin loses no digits), sums of 128 terms in FP32, the sums of those in
// FP64.  A target whose sum lies within FLD_SIDE_EPS sum_j w_j/r_j of the threshold (every rounding
// error above is below a tenth of that), or that has a node at a distance whose square is near the ends
// of FP32's range (or beyond, or zero: FLD_R2_MIN, FLD_R2_MAX), is summed again in FP64.  0.1 ms for 3001 targets and 16384 nodes, where one FP64
// thread per target took 10.4 ms.
#define FLD_SIDE_EPS 1e-4f
#define FLD_R2_MIN 1e-30f
#define FLD_R2_MAX 1e30f
struct SideSlot {
  float xh, xl, yh, yl, nx, ny, w;
};

__global__ void __launch_bounds__(FLD_THREADS)
    k_field_side(DevGeom g, const double* __restrict__ tx, const double* __restrict__ ty, int64_t nt, int64_t jspan,
                 double2* __restrict__ part) {
  __shared__ SideSlot sj[FLD_THREADS];
  const int64_t t = (int64_t)blockIdx.x * FLD_THREADS + threadIdx.x;
  const double px = t < nt ? tx[t] : 0.0, py = t < nt ? ty[t] : 0.0;
  const double x0 = g.x[0], y0 = g.y[0], qx = px - x0, qy = py - y0;
  const float pxh = (float)qx, pyh = (float)qy, pxl = (float)(qx - (double)pxh), pyl = (float)(qy - (double)pyh);
  const int64_t j0 = (int64_t)blockIdx.y * jspan, j1 = min(g.n, j0 + jspan);
  double acc = 0.0, mag = 0.0;
  for (int64_t jc = j0; jc < j1; jc += FLD_THREADS) {
    __syncthreads();
    const int64_t j = jc + threadIdx.x;
    if (j < j1) {
      SideSlot& s = sj[threadIdx.x];
      const double x = g.x[j] - x0, y = g.y[j] - y0;
      s.xh = (float)x;
      s.xl = (float)(x - (double)s.xh);
      s.yh = (float)y;
      s.yl = (float)(y - (double)s.yh);
      s.nx = (float)g.nx[j];
      s.ny = (float)g.ny[j];
      s.w = (float)g.w[j];
    }
    __syncthreads();
    const int nj = (int)min((int64_t)FLD_THREADS, j1 - jc);
    float a = 0.0f, m = 0.0f;
    for (int jj = 0; jj < nj; ++jj) {
      const SideSlot& s = sj[jj];
      const float dx = (pxh - s.xh) + (pxl - s.xl), dy = (pyh - s.yh) + (pyl - s.yl);
      const float r2 = fmaf(dx, dx, dy * dy);
      const float ir = rsqrtf(r2);
      const float wr = s.w * ir;
      a = fmaf(wr * ir, fmaf(dx, s.nx, dy * s.ny), a);
      // an infinite m leaves the decision to the FP64 sum, whatever became of the term
      m += r2 > FLD_R2_MIN && r2 < FLD_R2_MAX ? fabsf(wr) : __int_as_float(0x7F800000);
    }
    acc += (double)a;
    mag += (double)m;
  }
  if (t < nt) part[(int64_t)blockIdx.y * nt + t] = make_double2(acc, mag);
}

// side[t] = 1 inside, 0 outside: a warp per target, so that targets summed again in FP64 spread over the GPU
// (500 targets on the nodes of a curve of 500: a CTA per 128 targets took as long as the field itself).
__global__ void __launch_bounds__(FLD_THREADS)
    k_field_side_finish(DevGeom g, const double* __restrict__ tx, const double* __restrict__ ty, int64_t nt,
                        int nsplit, const double2* __restrict__ part, int8_t* __restrict__ side) {
  const int lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * (FLD_THREADS / 32) + (threadIdx.x >> 5);
  if (t >= nt) return;
  auto sum = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
  };
  double acc = 0.0, mag = 0.0;
  for (int p = lane; p < nsplit; p += 32) {
    const double2 v = part[(int64_t)p * nt + t];
    acc += v.x;
    mag += v.y;
  }
  acc = sum(acc);
  mag = sum(mag);
  const double off = fabs(acc + WSBM_PI);  // 2 pi |sum - 1/2|
  if (!(off > (double)FLD_SIDE_EPS * mag)) {  // also an infinite or NaN mag
    const double px = tx[t], py = ty[t];
    acc = 0.0;
    for (int64_t j = lane; j < g.n; j += 32) {
      const double dx = px - g.x[j], dy = py - g.y[j];
      const double r2 = dx * dx + dy * dy;
      if (r2 > 0.0) acc += g.w[j] * (dx * g.nx[j] + dy * g.ny[j]) / r2;
    }
    acc = sum(acc);
  }
  if (lane == 0) side[t] = (-acc / (2.0 * WSBM_PI)) > 0.5 ? 1 : 0;
}

// Partial sums over the sources [j0, j1) of CTA row blockIdx.y, for the nc <= NR right-hand sides
// starting at column c0.  part: nsplit x nt x NR complex128.  Bound by the FP64 pipe: 31 operations
// a pair (Hankel values in fixed point, one reciprocal square root each for 1/r and the amplitude,
// the side's signs and constants folded into two factors) and 8 per right-hand side.  16384 nodes, 3001
// targets, 8 columns: 8.5 ms (25 ms in two launches of 4 columns with FP64 Hankel values).
template <int NR>
__global__ void __launch_bounds__(FLD_THREADS)
    k_field(DevGeom g, Phys ph, const double2* __restrict__ u, const double2* __restrict__ q, int nc, int c0,
            const double* __restrict__ tx, const double* __restrict__ ty, int64_t nt,
            const int8_t* __restrict__ side, int64_t jspan, double2* __restrict__ part) {
  __shared__ HkTables T;
  __shared__ FldSlot sj[FLD_THREADS];
  __shared__ double2 su[NR][FLD_THREADS], sq[NR][FLD_THREADS];
  hk_stage_tables(&T);
  const int64_t N = g.n;
  const int64_t t = (int64_t)blockIdx.x * FLD_THREADS + threadIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * jspan, j1 = min(N, j0 + jspan);
  const bool valid = t < nt;
  const double px = valid ? tx[t] : 0.0, py = valid ? ty[t] : 0.0;
  const bool in = valid && side[t] != 0;
  const double k = in ? ph.k1 : ph.k0, ik = in ? ph.inv_k1 : ph.inv_k0;
  // w G = (i w/4) H0, times eps1 inside, -eps0 outside;  w dG/dn_y = (i k w/4) H1 (d.n)/r, times
  // -1 inside, 1 outside
  const double ea = 0.25 * (in ? ph.eps1 : -ph.eps0), eb = (in ? -0.25 : 0.25) * k;
  double2 acc[NR];
#pragma unroll
  for (int c = 0; c < NR; ++c) acc[c] = make_double2(0.0, 0.0);
  for (int64_t jc = j0; jc < j1; jc += FLD_THREADS) {
    __syncthreads();
    {
      int64_t j = jc + threadIdx.x;
      if (j < j1) {
        FldSlot& s = sj[threadIdx.x];
        s.x = g.x[j];
        s.y = g.y[j];
        s.nx = g.nx[j];
        s.ny = g.ny[j];
        s.w = g.w[j];
#pragma unroll
        for (int c = 0; c < NR; ++c) {
          su[c][threadIdx.x] = c < nc ? u[(int64_t)(c0 + c) * N + j] : make_double2(0.0, 0.0);
          sq[c][threadIdx.x] = c < nc ? q[(int64_t)(c0 + c) * N + j] : make_double2(0.0, 0.0);
        }
      }
    }
    __syncthreads();
    if (!valid) continue;
    const int nj = (int)min((int64_t)FLD_THREADS, j1 - jc);
#pragma unroll 1
    for (int jj = 0; jj < nj; ++jj) {
      // keep the Hankel tables in shared memory: no hoisting of their loads out of the loop
      asm volatile("" ::: "memory");
      const FldSlot& s = sj[jj];
      const double dx = px - s.x, dy = py - s.y;
      const double r2 = pair_r2(dx, dy);
      if (r2 == 0.0) continue;
      const double rs = rsqrt3_any(r2);  // 1/r
      const double z = k * sqrt_from(r2, rs);
      const double dn = fma(dx, s.nx, dy * s.ny) * rs;
      const int zhi = __double2hiint(z);
      double2 G, D;
      if (zhi >= HK_SERIES_HI && zhi < HX_Z_HI_WORD) {
        HxUnit h;
        hankel_fixed(T.near_, z, rs * ik, h);
        const double wa = s.w * (WSBM_SQRT_2_OVER_PI * rsqrt3(z));
        const double sg = ea * wa, sd = eb * wa * dn;
        G = make_double2(-sg * h.i0, sg * h.r0);
        D = make_double2(-sd * h.i1, sd * h.r1);
      } else {
        Hk h;
        hankel_fp64_rs<false>(T, z, rsqrt(z), h);
        const double sg = ea * s.w, sd = eb * s.w * dn;
        G = make_double2(-sg * h.h0i, sg * h.h0r);
        D = make_double2(-sd * h.h1i, sd * h.h1r);
      }
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        const double2 uu = su[c][jj], qq = sq[c][jj];
        acc[c].x = fma(G.x, qq.x, fma(-G.y, qq.y, fma(D.x, uu.x, fma(-D.y, uu.y, acc[c].x))));
        acc[c].y = fma(G.x, qq.y, fma(G.y, qq.x, fma(D.x, uu.y, fma(D.y, uu.x, acc[c].y))));
      }
    }
  }
  if (valid) {
#pragma unroll
    for (int c = 0; c < NR; ++c) part[((int64_t)blockIdx.y * nt + t) * NR + c] = acc[c];
  }
}

__global__ void k_field_reduce(int64_t nt, int nsplit, int nc, int nr, int c0, const double2* __restrict__ part,
                               double2* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nt * nc;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = e / nc;
    const int c = (int)(e % nc);
    double2 s = make_double2(0.0, 0.0);
    for (int p = 0; p < nsplit; ++p) {
      double2 v = part[((int64_t)p * nt + t) * nr + c];
      s.x += v.x;
      s.y += v.y;
    }
    out[(int64_t)(c0 + c) * nt + t] = s;
  }
}

int grid_cap(int64_t blocks) {
  const int64_t cap = (int64_t)wsbm_sm_count() * 16;
  return (int)(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

}  // namespace

int wsbm_phys_from_params(const wsbm_params* p, Phys* ph);
int wsbm_geom_check(const wsbm_geom* g);
DevGeom wsbm_devgeom(const wsbm_geom* g);

extern "C" int wsbm_field(const wsbm_geom* g, const wsbm_params* p, const void* u, const void* q,
                          int32_t nrhs, const double* tx, const double* ty, int64_t nt, void* out,
                          int8_t* inside, void* stream) {
  int rc = wsbm_geom_check(g);
  if (rc) return rc;
  Phys ph;
  if ((rc = wsbm_phys_from_params(p, &ph))) return rc;
  if (nrhs < 1 || nt < 0 || !u || !q || (nt > 0 && (!tx || !ty || !out || !inside)))
    return WSBM_ERR_INVALID_ARG;
  if (nt == 0) return WSBM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t N = g->n;
  const int64_t nti = (nt + FLD_THREADS - 1) / FLD_THREADS;
  // the split, hence a column's rounding, depends on N and the targets alone and not on how many columns
  // come along: at least 128 sources a CTA
  const int64_t want = (int64_t)wsbm_sm_count() * FLD_WANT;
  int64_t nsplit = std::max<int64_t>(1, std::min<int64_t>((want + nti - 1) / nti, (N + 127) / 128));
  const int64_t jspan = ((N + nsplit - 1) / nsplit + FLD_THREADS - 1) / FLD_THREADS * FLD_THREADS;
  nsplit = (N + jspan - 1) / jspan;
  WsbmScratch scr(st);
  double2* part = nullptr;
  int nr = nrhs > 4 ? 8 : (nrhs > 2 ? 4 : nrhs);  // right-hand sides per launch, fewer where the scratch is short
  while ((rc = scr.get((size_t)nsplit * nt * nr * sizeof(double2), (void**)&part)) == WSBM_ERR_OOM && nr > 1) nr /= 2;
  if (rc) return rc;
  DevGeom dg = wsbm_devgeom(g);
  const dim3 grid((unsigned)nti, (unsigned)nsplit);
  k_field_side<<<grid, FLD_THREADS, 0, st>>>(dg, tx, ty, nt, jspan, part);
  k_field_side_finish<<<(unsigned)((nt + FLD_THREADS / 32 - 1) / (FLD_THREADS / 32)), FLD_THREADS, 0, st>>>(dg, tx, ty, nt, (int)nsplit, part, inside);
  wsbm_count_launches(2);
  const double2 *cu = (const double2*)u, *cq = (const double2*)q;
  for (int c0 = 0; c0 < nrhs; c0 += nr) {
    const int nc = std::min(nr, nrhs - c0);
    if (nr == 8)
      k_field<8><<<grid, FLD_THREADS, 0, st>>>(dg, ph, cu, cq, nc, c0, tx, ty, nt, inside, jspan, part);
    else if (nr == 4)
      k_field<4><<<grid, FLD_THREADS, 0, st>>>(dg, ph, cu, cq, nc, c0, tx, ty, nt, inside, jspan, part);
    else if (nr == 2)
      k_field<2><<<grid, FLD_THREADS, 0, st>>>(dg, ph, cu, cq, nc, c0, tx, ty, nt, inside, jspan, part);
    else
      k_field<1><<<grid, FLD_THREADS, 0, st>>>(dg, ph, cu, cq, nc, c0, tx, ty, nt, inside, jspan, part);
    k_field_reduce<<<grid_cap((nt * nc + 255) / 256), 256, 0, st>>>(nt, (int)nsplit, nc, nr, c0, part, (double2*)out);
    wsbm_count_launches(2);
  }
  return cudaGetLastError() == cudaSuccess ? WSBM_OK : WSBM_ERR_CUDA;
}
