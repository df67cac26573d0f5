// Matrix-free products with the full WSBM Nystrom matrix (no storage): y = A x and y = A^T x.
#include <math.h>

#include "entry_blocks.cuh"

// Matrix-free product y = A x (TRANS: y = A^T x) over every node pair (dense, O(N^2) pair
// evaluations; used for residuals and iterative refinement of HSS and adjoint solutions).
// Thread = output node i; CTA row blockIdx.y covers the other nodes [j0, j1); per-split
// partial sums, reduced in a fixed order by k_matvec_reduce.  Vectors in paper order.
#define MV_THREADS 128
#define MV_FLUSH 16  // divides MV_THREADS
// CTAs per SM.  N = 16384, one and eight columns: 45.5 and 96.5 ms, 47.8 and 95.5 with 16 (a last wave that
// is nearly empty), 48.4 and 101.7 with 8
#define MV_WANT 32
template <int NR>
struct MvSlot {
  double x, y, nx, ny, w;
  double2 u[NR], q[NR];
};

// nr <= NR columns c0 .. c0 + nr - 1 of x (column stride 2N; NR = 1, 2, 4 or 8 share each pair's
// entries, absent ones are zero); partial sums of column r of split s at part[(s * NR + r) * 2N +
// row].  Bound by the FP64 pipe: 71 operations a pair for the entries and 16 per column, so 8
// columns at once take 199 where two passes of 4 take 270.
// Each of a pair's four products rounds at the size of the running sum, so the running sums are short:
// every MV_FLUSH pairs they go into the partial sums in memory and begin again.  Error of y against long
// double, 1000-node star, 4 columns: 3.4e-16 (4.5e-16 with the four products summed first, which takes
// 20 operations a column; 7.7e-16 with one running sum).
template <bool TRANS, int NR>
__global__ void __launch_bounds__(MV_THREADS)
    k_matvec(DevGeom g, Phys ph, const double2* __restrict__ xin, int nr, int64_t jspan,
             double2* __restrict__ part) {
  __shared__ HkTables T;
  __shared__ MvSlot<NR> sj[MV_THREADS];
  hk_stage_tables(&T);
  const int64_t N = g.n;
  const int64_t i = (int64_t)blockIdx.x * MV_THREADS + threadIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * jspan;
  const int64_t j1 = min(N, j0 + jspan);
  const bool valid = i < N;
  double xi = 0, yi = 0, nxi = 0, nyi = 0, wi = 0, ki = 0;
  if (valid) {
    xi = g.x[i];
    yi = g.y[i];
    nxi = g.nx[i];
    nyi = g.ny[i];
    wi = g.w[i];
    ki = g.kappa[i];
  }
  double2 a0[NR], a1[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) a0[r] = a1[r] = make_double2(0.0, 0.0);
  for (int64_t jc = j0; jc < j1; jc += MV_THREADS) {
    __syncthreads();
    {
      int64_t j = jc + threadIdx.x;
      if (j < j1) {
        MvSlot<NR>& s = sj[threadIdx.x];
        s.x = g.x[j];
        s.y = g.y[j];
        s.nx = g.nx[j];
        s.ny = g.ny[j];
        s.w = g.w[j];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const bool on = r < nr;
          s.u[r] = on ? xin[(int64_t)r * 2 * N + j] : make_double2(0.0, 0.0);
          s.q[r] = on ? xin[(int64_t)r * 2 * N + N + j] : make_double2(0.0, 0.0);
        }
      }
    }
    __syncthreads();
    const unsigned mask = __ballot_sync(0xFFFFFFFFu, valid);
    if (!valid) continue;
    const int nj = (int)min((int64_t)MV_THREADS, j1 - jc);
#pragma unroll 1
    for (int jj = 0; jj < nj; ++jj) {
      // keep the Hankel tables in shared memory: no hoisting of their loads out of the loop
      asm volatile("" ::: "memory");
      const MvSlot<NR>& s = sj[jj];
      double2 e[2][2];
      // block (i, j): row node i, column node j; TRANS: block (j, i), applied transposed.  A warp with pairs
      // out of the fixed-point range takes the general path for all of its pairs: half the way through both
      // would cost more (64 nodes, 15 a wavelength: 983 us, now 870; 2000 nodes: 1766, 1637)
      const bool diag = jc + jj == i;
      const double sx = TRANS ? s.x : xi, sy = TRANS ? s.y : yi, tx = TRANS ? xi : s.x, ty = TRANS ? yi : s.y;
      const double snx = TRANS ? s.nx : nxi, sny = TRANS ? s.ny : nyi, tnx = TRANS ? nxi : s.nx, tny = TRANS ? nyi : s.ny;
      const double w = TRANS ? wi : s.w, dx = __dsub_rn(sx, tx), dy = __dsub_rn(sy, ty), r2 = pair_r2(dx, dy);
      const bool fixed = __all_sync(mask, diag || pair_is_fixed(ph, r2));
      if (diag) {
        block_diag(ph, wi, ki, e);
      } else if (fixed) {
        block_fixed(T, ph, dx, dy, r2, snx, sny, tnx, tny, w, e);
      } else {
        PairGeom G;
        pair_geom(sx, sy, snx, sny, tx, ty, tnx, tny, ph, G);
        block_offdiag(T, ph, G, w, e);
      }
      if (TRANS) {
        double2 t = e[0][1];
        e[0][1] = e[1][0];
        e[1][0] = t;
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double2 u = s.u[r], q = s.q[r];
        a0[r].x = fma(e[0][0].x, u.x, fma(-e[0][0].y, u.y, fma(e[0][1].x, q.x, fma(-e[0][1].y, q.y, a0[r].x))));
        a0[r].y = fma(e[0][0].x, u.y, fma(e[0][0].y, u.x, fma(e[0][1].x, q.y, fma(e[0][1].y, q.x, a0[r].y))));
        a1[r].x = fma(e[1][0].x, u.x, fma(-e[1][0].y, u.y, fma(e[1][1].x, q.x, fma(-e[1][1].y, q.y, a1[r].x))));
        a1[r].y = fma(e[1][0].x, u.y, fma(e[1][0].y, u.x, fma(e[1][1].x, q.y, fma(e[1][1].y, q.x, a1[r].y))));
      }
      if (((jj + 1) & (MV_FLUSH - 1)) != 0 && jj + 1 < nj) continue;
      const bool first = jc == j0 && jj < MV_FLUSH;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (r >= nr) break;
        double2* pr = part + ((int64_t)blockIdx.y * NR + r) * 2 * N + i;
        const double2 b0 = first ? make_double2(0.0, 0.0) : pr[0], b1 = first ? make_double2(0.0, 0.0) : pr[N];
        pr[0] = make_double2(b0.x + a0[r].x, b0.y + a0[r].y);
        pr[N] = make_double2(b1.x + a1[r].x, b1.y + a1[r].y);
        a0[r] = a1[r] = make_double2(0.0, 0.0);
      }
    }
  }
}

// y[:, r] = sum over the splits, in split order, for the nr columns of one launch.
__global__ void k_matvec_reduce(int64_t N, int nsplit, int nr, int NR, const double2* __restrict__ part,
                                double2* __restrict__ y) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 2 * N * nr;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / (2 * N), row = e % (2 * N);
    double2 s = make_double2(0.0, 0.0);
    for (int t = 0; t < nsplit; ++t) {
      double2 v = part[((int64_t)t * NR + r) * 2 * N + row];
      s.x += v.x;
      s.y += v.y;
    }
    y[r * 2 * N + row] = s;
  }
}

static int grid_for(int64_t blocks) {
  const int64_t cap = (int64_t)wsbm_sm_count() * 16;
  return (int)(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

int wsbm_phys_from_params(const wsbm_params* p, Phys* ph);
int wsbm_geom_check(const wsbm_geom* g);
DevGeom wsbm_devgeom(const wsbm_geom* g);

extern "C" int wsbm_matvec(const wsbm_geom* g, const wsbm_params* p, int32_t trans, const void* x,
                           int32_t nrhs, void* y, void* stream) {
  int rc = wsbm_geom_check(g);
  if (rc) return rc;
  Phys ph;
  if ((rc = wsbm_phys_from_params(p, &ph))) return rc;
  if (p->formulation != WSBM_FORM_WSBM) return WSBM_ERR_INVALID_ARG;  // eq. (weakly_bm) only
  if ((trans != 0 && trans != 1) || nrhs < 0 || (nrhs > 0 && (!x || !y))) return WSBM_ERR_INVALID_ARG;
  if (nrhs == 0) return WSBM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t N = g->n;
  const int64_t nti = (N + MV_THREADS - 1) / MV_THREADS;
  // the split, hence a column's rounding, depends on N alone and not on how many columns come along
  const int64_t want = (int64_t)wsbm_sm_count() * MV_WANT;
  int64_t nsplit = (want + nti - 1) / nti;
  if (nsplit < 1) nsplit = 1;
  if (nsplit > nti) nsplit = nti;
  const int64_t jspan = (N + nsplit - 1) / nsplit;
  nsplit = (N + jspan - 1) / jspan;
  WsbmScratch scr(st);
  double2* part = nullptr;
  int NR = nrhs > 4 ? 8 : (nrhs > 2 ? 4 : nrhs);  // columns of one launch, fewer where the scratch is short
  while ((rc = scr.get((size_t)nsplit * NR * 2 * N * sizeof(double2), (void**)&part)) == WSBM_ERR_OOM && NR > 1) NR /= 2;
  if (rc) return rc;
  const auto kern = trans ? (NR == 8 ? k_matvec<true, 8> : NR == 4 ? k_matvec<true, 4> : NR == 2 ? k_matvec<true, 2> : k_matvec<true, 1>)
                          : (NR == 8 ? k_matvec<false, 8> : NR == 4 ? k_matvec<false, 4> : NR == 2 ? k_matvec<false, 2> : k_matvec<false, 1>);
  DevGeom dg = wsbm_devgeom(g);
  for (int c = 0; c < nrhs; c += NR) {
    const int nr = nrhs - c < NR ? nrhs - c : NR;
    const double2* xc = (const double2*)x + (int64_t)c * 2 * N;
    kern<<<dim3((unsigned)nti, (unsigned)nsplit), MV_THREADS, 0, st>>>(dg, ph, xc, nr, jspan, part);
    int64_t blocks = (2 * N * nr + 255) / 256;
    k_matvec_reduce<<<grid_for(blocks), 256, 0, st>>>(N, (int)nsplit, nr, NR, part, (double2*)y + (int64_t)c * 2 * N);
    wsbm_count_launches(2);
    if (cudaGetLastError() != cudaSuccess) return WSBM_ERR_CUDA;
  }
  return WSBM_OK;
}
