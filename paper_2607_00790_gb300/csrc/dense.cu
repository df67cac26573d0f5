// Batched dense complex128 linear algebra for the HSS factor (Martinsson-Rokhlin solver,
// Sec. III): blocked LU with partial pivoting, blocked triangular solves, complex GEMM and a
// column-pivoted Householder QR for the interpolative decompositions.
//
// Every routine works on a batch of column-major matrices of different sizes described by
// device arrays.  Blocked algorithms step through panels of WSBM_NB columns on the host; each
// step launches one kernel over the whole batch (matrices that are already finished skip).
// The O(n^3) work is in the GEMM kernel, which tiles every matrix of the batch over many CTAs.
#include <math.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "cplx.cuh"
#include "dense.h"
#include "rowswap.cuh"
#include "tri.cuh"

#define GT 32  // GEMM tile (GT x GT outputs per CTA)
#define GK 16  // GEMM k-chunk

// --------------------------------------------------------------------------- GEMM ----
// C[m x n] = alpha * A[m x k] * B[k x n] + beta * C, one GT x GT tile of C.
template <bool TA>
__device__ void gemm_tile(int m, int n, int k, const double2* __restrict__ A, int64_t lda,
                          const double2* __restrict__ B, int64_t ldb, double2* C, int64_t ldc,
                          double2 alpha, double2 beta, int tm, int tn) {
  __shared__ double2 sA[GK][GT + 1];
  __shared__ double2 sB[GK][GT + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;  // 256 threads: 16 x 16, 2x2 each
  const int i0 = tm * GT, j0 = tn * GT;
  double2 acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = make_double2(0.0, 0.0);
  for (int kk = 0; kk < k; kk += GK) {
    __syncthreads();
    for (int t = threadIdx.x; t < GK * GT; t += blockDim.x) {
      int r = t % GT, c = t / GT;  // A: row r of the tile, k index c
      int gi = i0 + r, gk = kk + c;
      sA[c][r] = (gi < m && gk < k) ? A[TA ? gk + (int64_t)gi * lda : gi + (int64_t)gk * lda]
                                    : make_double2(0.0, 0.0);
      int br = t % GK, bc = t / GK;  // B: k index br, column bc
      int gk2 = kk + br, gj = j0 + bc;
      sB[br][bc] = (gk2 < k && gj < n) ? B[gk2 + (int64_t)gj * ldb] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < GK; ++c) {
      double2 a0 = sA[c][tx], a1 = sA[c][tx + 16];
      double2 b0 = sB[c][ty], b1 = sB[c][ty + 16];
      acc[0][0] = cfma(a0, b0, acc[0][0]);
      acc[1][0] = cfma(a1, b0, acc[1][0]);
      acc[0][1] = cfma(a0, b1, acc[0][1]);
      acc[1][1] = cfma(a1, b1, acc[1][1]);
    }
  }
  const bool beta0 = beta.x == 0.0 && beta.y == 0.0;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      int gi = i0 + tx + 16 * a, gj = j0 + ty + 16 * b;
      if (gi < m && gj < n) {
        double2* p = C + gi + (int64_t)gj * ldc;
        double2 v = cmul(alpha, acc[a][b]);
        *p = beta0 ? v : cfma(beta, *p, v);
      }
    }
}

__global__ void __launch_bounds__(256) k_gemm(const GemmDesc* __restrict__ d, int nbatch) {
  const GemmDesc g = d[blockIdx.y];
  int ntm = (g.m + GT - 1) / GT, ntn = (g.n + GT - 1) / GT;
  for (int t = blockIdx.x; t < ntm * ntn; t += gridDim.x) {
    if (g.ta)
      gemm_tile<true>(g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.C, g.ldc, g.alpha, g.beta, t % ntm, t / ntm);
    else
      gemm_tile<false>(g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.C, g.ldc, g.alpha, g.beta, t % ntm, t / ntm);
  }
}

// The same for a few columns (n <= GEMM_FEW), a column per blockIdx.z: a warp has 16 rows, a lane one
// real component of one, so no lane works on columns that are not there and a step of the sum costs two
// FP64 instructions a warp (64 clocks each on its sub-partition) in place of 32.  Operands come from
// L1/L2, GF_K steps ahead of the sum.  The order of operations is k_gemm's.
#define GEMM_FEW 8
#define GF_K 8
__global__ void __launch_bounds__(128) k_gemm_few(const GemmDesc* __restrict__ d) {
  const GemmDesc g = d[blockIdx.y];
  const int lane = threadIdx.x & 31, part = lane & 1, c = blockIdx.z, neg = part ? 0 : (int)0x80000000;
  if (c >= g.n) return;
  const double* B = (const double*)(g.B + (int64_t)c * g.ldb);
  const int64_t sa = g.ta ? 1 : g.lda;
  for (int r0 = blockIdx.x * 64 + (threadIdx.x >> 5) * 16; r0 < g.m; r0 += gridDim.x * 64) {
    const int i = r0 + (lane >> 1);
    const double2* A = g.A + (int64_t)min(i, g.m - 1) * (g.ta ? g.lda : 1);
    double acc = 0.0;
    double2 a[GF_K], na[GF_K];
    double own[GF_K], oth[GF_K], nown[GF_K], noth[GF_K];
    auto load = [&](int t0, double2(&x)[GF_K], double(&u)[GF_K], double(&v)[GF_K]) {
#pragma unroll
      for (int t = 0; t < GF_K; ++t) {
        const bool in = t0 + t < g.k;
        x[t] = in ? A[(t0 + t) * sa] : make_double2(0.0, 0.0);
        u[t] = in ? B[2 * (t0 + t) + part] : 0.0;
        v[t] = in ? B[2 * (t0 + t) + 1 - part] : 0.0;
      }
    };
    load(0, a, own, oth);
    for (int t0 = 0; t0 < g.k; t0 += GF_K) {
      load(t0 + GF_K, na, nown, noth);
#pragma unroll
      for (int t = 0; t < GF_K; ++t) {  // cfma, one component
        const double ay = __hiloint2double(__double2hiint(a[t].y) ^ neg, __double2loint(a[t].y));
        acc = fma(a[t].x, own[t], fma(ay, oth[t], acc));
        a[t] = na[t];
        own[t] = nown[t];
        oth[t] = noth[t];
      }
    }
    // the complex epilogue of k_gemm: each lane of a pair forms it and keeps its component
    const bool in = i < g.m, beta0 = g.beta.x == 0.0 && g.beta.y == 0.0;
    double* p = (double*)(g.C + i + (int64_t)c * g.ldc) + part;
    const double old = in && !beta0 ? *p : 0.0;
    const double acc2 = __shfl_xor_sync(0xFFFFFFFFu, acc, 1), old2 = __shfl_xor_sync(0xFFFFFFFFu, old, 1);
    double2 v = cmul(g.alpha, part ? make_double2(acc2, acc) : make_double2(acc, acc2));
    if (!beta0) v = cfma(g.beta, part ? make_double2(old2, old) : make_double2(old, old2), v);
    if (in) *p = part ? v.y : v.x;
  }
}

// LU trailing update at panel j0 (width jb): A22 -= A21 * A12.
__global__ void __launch_bounds__(256) k_lu_update(const LuDesc* __restrict__ d, int j0, int jb) {
  const LuDesc q = d[blockIdx.y];
  int e = j0 + jb;
  if (e >= q.n) return;
  int m = q.n - e;
  int nt = (m + GT - 1) / GT;
  const double2 one = make_double2(1.0, 0.0), mone = make_double2(-1.0, 0.0);
  int kb = min(jb, q.n - j0);
  for (int t = blockIdx.x; t < nt * nt; t += gridDim.x)
    gemm_tile<false>(m, m, kb, q.A + e + (int64_t)j0 * q.lda, q.lda, q.A + j0 + (int64_t)e * q.lda, q.lda,
              q.A + e + (int64_t)e * q.lda, q.lda, mone, one, t % nt, t / nt);
}

// ------------------------------------------------------------------- LU panel ----
// Factor columns [j0, j0+jb) (jb <= LUP_W) of rows [j0, n) in place with partial pivoting; row swaps are
// applied inside the panel only (k_laswp applies them elsewhere).  One CTA per matrix.
// A sub-partition takes 64 clocks for every FP64 instruction of a warp, so what every warp would repeat
// is kept off that pipe: the moduli are compared by their bits, one warp takes the reciprocal (beside
// the row swap of the others).  A thread scales its row's multiplier, updates the row eight columns at
// a time (their loads in flight together) and brings the next column's candidate: two barriers a column.
// 64 columns of box matrices, one matrix per SM: 850 us before, 530 us; bound by FP64 on that SM.
#define LUP_W 64
#define LUP_C 8
__global__ void __launch_bounds__(256) k_lu_panel(const LuDesc* __restrict__ d, int j0, int jb,
                                                  int* __restrict__ info) {
  const LuDesc q = d[blockIdx.x];
  if (j0 >= q.n) return;
  const int n = q.n;
  const int je = min(j0 + jb, n);
  double2* A = q.A;
  const int64_t lda = q.lda;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ long long skey[8];
  __shared__ int sidx[8];
  __shared__ double2 su[LUP_W], sinv;
  auto key = [](double2 v) {  // |v|^2 as an integer of the same order; NaN never wins
    const long long b = __double_as_longlong(cabs2(v));
    return b > 0x7ff0000000000000ll ? -1ll : b;
  };
  long long best = -1;
  int bi = j0;
  for (int i = j0 + tid; i < n; i += 256) {
    const long long v = key(A[i + (int64_t)j0 * lda]);
    if (v > best) {
      best = v;
      bi = i;
    }
  }
  for (int j = j0; j < je; ++j) {
    // pivot: the largest modulus, first row on ties
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    if (lane == 0) {
      skey[warp] = best;
      sidx[warp] = bi;
    }
    __syncthreads();
    best = skey[0];
    int p = sidx[0];
#pragma unroll
    for (int w = 1; w < 8; ++w)
      if (skey[w] > best || (skey[w] == best && sidx[w] < p)) {
        best = skey[w];
        p = sidx[w];
      }
    if (warp == 0) {  // column j: its swap and the reciprocal
      const double2 v = A[p + (int64_t)j * lda], o = A[j + (int64_t)j * lda];
      __syncwarp();
      if (lane == 0) {
        q.piv[j] = p;
        if (best == 0 && info) info[blockIdx.x] = j + 1;  // exactly singular
        if (p != j) {
          A[j + (int64_t)j * lda] = v;
          A[p + (int64_t)j * lda] = o;
        }
        sinv = (v.x == 0.0 && v.y == 0.0) ? make_double2(0.0, 0.0) : cdiv(make_double2(1.0, 0.0), v);
      }
    } else {
      for (int c = j0 + tid - 32; c < je; c += 224) {
        if (c == j) continue;
        const double2 v = A[p + (int64_t)c * lda];
        if (p != j) {
          A[p + (int64_t)c * lda] = A[j + (int64_t)c * lda];
          A[j + (int64_t)c * lda] = v;
        }
        su[c - j0] = v;
      }
    }
    __syncthreads();
    const double2 inv = sinv;
    best = -1;
    bi = j + 1;
    for (int i = j + 1 + tid; i < n; i += 256) {
      double2* r = A + i;
      const double2 l = cmul(r[(int64_t)j * lda], inv);
      r[(int64_t)j * lda] = l;
      for (int c = j + 1; c < je; c += LUP_C) {
        double2 x[LUP_C];
#pragma unroll
        for (int t = 0; t < LUP_C; ++t)
          if (c + t < je) x[t] = r[(int64_t)(c + t) * lda];
#pragma unroll
        for (int t = 0; t < LUP_C; ++t)
          if (c + t < je) {
            x[t] = cfms(l, su[c + t - j0], x[t]);
            r[(int64_t)(c + t) * lda] = x[t];
          }
        if (c == j + 1) {
          const long long v = key(x[0]);
          if (v > best) {
            best = v;
            bi = i;
          }
        }
      }
    }
  }
}

// Apply the row interchanges of panel [j0, j0+jb) to the columns outside the panel.
__global__ void k_laswp(const LuDesc* __restrict__ d, int j0, int jb) {
  const LuDesc q = d[blockIdx.y];
  if (j0 >= q.n) return;
  const int je = min(j0 + jb, q.n);
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < q.n; c += gridDim.x * blockDim.x) {
    if (c >= j0 && c < je) continue;
    double2* col = q.A + (int64_t)c * q.lda;
    for (int j = j0; j < je; ++j) {
      int p = q.piv[j];
      if (p != j) {
        double2 t = col[j];
        col[j] = col[p];
        col[p] = t;
      }
    }
  }
}

// A12 = L11^-1 A12 for the block row of panel [j0, j0+jb) (unit lower L11), columns >= j0+jb.
__global__ void k_lu_trsm_row(const LuDesc* __restrict__ d, int j0, int jb) {
  const LuDesc q = d[blockIdx.y];
  const int je = min(j0 + jb, q.n);
  if (je >= q.n) return;
  for (int c = je + blockIdx.x * blockDim.x + threadIdx.x; c < q.n; c += gridDim.x * blockDim.x) {
    double2* col = q.A + (int64_t)c * q.lda;
    for (int i = j0 + 1; i < je; ++i) {
      double2 s = col[i];
      for (int t = j0; t < i; ++t) s = cfms(q.A[i + (int64_t)t * q.lda], col[t], s);
      col[i] = s;
    }
  }
}

// ------------------------------------------------------------- triangular solves ----
// B <- op(T)^-1 B for a diagonal block [j0, j0 + jb) of T (jb <= 32; lower unit or upper non-unit).
// The block is staged as a lower triangle S (rows and columns reversed for a backward solve) with
// the reciprocals of its diagonal, zero rows and columns beyond the matrix.
struct TrsmStage {
  double2 S[32][33];  // S[t][i]: column t, row i of the triangle
  double2 inv[32];
};
__device__ __forceinline__ double2 trsm_elem(const TrsmDesc& q, int j0, int b, int e) {
  const int a = e & 31, c = e >> 5;  // element (a, c) of the stored block
  return a < b && c < b ? q.T[(j0 + a) + (int64_t)(j0 + c) * q.ldt] : make_double2(0.0, 0.0);
}
__device__ __forceinline__ void trsm_put(TrsmStage& D, const TrsmDesc& q, int b, bool fwd, int e, double2 v) {
  const int a = e & 31, c = e >> 5;
  int i = q.trans ? c : a, t = q.trans ? a : c;
  if (a < b && c < b && !fwd) {
    i = b - 1 - i;
    t = b - 1 - t;
  }
  D.S[t][i] = v;  // read where i >= t only
}
// The reciprocals by one warp at once: a division in the loop above would run for the one diagonal lane
// of every pass, 32 times a block.  The columns are scaled by them, which takes a complex product out
// of every step of the chain: x_i = r_i / S_ii with r_i = b_i - sum (S_it / S_tt) r_t.
__device__ __forceinline__ void trsm_reciprocals(TrsmStage& D, int b, bool unit) {
  __syncthreads();
  const int i = threadIdx.x;
  if (unit) return;
  if (i < 32) D.inv[i] = i >= b ? make_double2(1.0, 0.0) : cdiv(make_double2(1.0, 0.0), D.S[i][i]);
  __syncthreads();
  for (int e = i; e < 32 * 32; e += blockDim.x)
    if ((e & 31) > (e >> 5)) D.S[e >> 5][e & 31] = cmul(D.S[e >> 5][e & 31], D.inv[e >> 5]);
  __syncthreads();
}
__device__ __forceinline__ void trsm_stage(TrsmStage& D, const TrsmDesc& q, int j0, int jb, bool fwd, bool unit) {
  const int b = min(jb, q.n - j0);
  for (int e0 = threadIdx.x; e0 < 32 * 32; e0 += 8 * blockDim.x) {  // blockDim.x = 64 or 128: 8 loads in flight
    double2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = trsm_elem(q, j0, b, e0 + k * blockDim.x);
#pragma unroll
    for (int k = 0; k < 8; ++k) trsm_put(D, q, b, fwd, e0 + k * blockDim.x, v[k]);
  }
  trsm_reciprocals(D, b, unit);
}

// One column of the staged block by a warp, row `lane` of the solve's order in each lane's x.
__device__ __forceinline__ double2 trsm_warp_column(const TrsmStage& D, int b, bool unit, double2 x) {
  const int lane = threadIdx.x & 31;
  for (int t = 0; t < b; ++t) {
    double2 xt;
    xt.x = __shfl_sync(0xFFFFFFFFu, x.x, t);
    xt.y = __shfl_sync(0xFFFFFFFFu, x.y, t);
    if (lane > t) x = cfms(D.S[t][lane], xt, x);
  }
  return unit ? x : cmul(x, D.inv[lane]);
}

// Few columns (up to a few thousand in the launch): one warp per column, its row `lane` in each
// lane's register: 32 dependent steps a block, where a thread per column takes 512.
__global__ void __launch_bounds__(128) k_trsm_diag_warp(const TrsmDesc* __restrict__ d, int j0, int jb, int fwd) {
  __shared__ TrsmStage D;
  const TrsmDesc q = d[blockIdx.y];
  const int lane = threadIdx.x & 31;
  if (j0 >= q.n || (int)blockIdx.x * 4 >= q.nrhs) return;
  const bool unit = (fwd != 0) != (q.trans != 0);  // L and L^T have a unit diagonal
  trsm_stage(D, q, j0, jb, fwd != 0, unit);
  const int b = min(jb, q.n - j0), row = j0 + (fwd ? lane : b - 1 - lane);
  for (int c = blockIdx.x * 4 + (threadIdx.x >> 5); c < q.nrhs; c += gridDim.x * 4) {
    double2* col = q.B + (int64_t)c * q.ldb;
    const double2 x = trsm_warp_column(D, b, unit, lane < b ? col[row] : make_double2(0.0, 0.0));
    if (lane < b) col[row] = x;
  }
}

// Many columns: one thread per column held in shared memory (the triangle's entries are broadcast
// reads), so every lane of the FP64 pipe works.  The same operations in the same order as above: a
// solution does not depend on how many columns share its launch.
#define TRSM_COLS 64
__global__ void __launch_bounds__(TRSM_COLS) k_trsm_diag(const TrsmDesc* __restrict__ d, int j0, int jb, int fwd) {
  __shared__ TrsmStage D;
  extern __shared__ double2 sx[];  // [32][TRSM_COLS + 1]: row i of the thread's column
  const TrsmDesc q = d[blockIdx.y];
  if (j0 >= q.n || (int)blockIdx.x * TRSM_COLS >= q.nrhs) return;
  const bool unit = (fwd != 0) != (q.trans != 0);
  trsm_stage(D, q, j0, jb, fwd != 0, unit);
  const int b = min(jb, q.n - j0), tid = threadIdx.x;
  for (int c0 = blockIdx.x * TRSM_COLS; c0 < q.nrhs; c0 += gridDim.x * TRSM_COLS) {
    const int nc = min(TRSM_COLS, q.nrhs - c0);
    __syncthreads();
    for (int e = tid; e < 32 * TRSM_COLS; e += TRSM_COLS) {
      const int i = e & 31, c = e >> 5;
      if (i < b && c < nc) sx[(fwd ? i : b - 1 - i) * (TRSM_COLS + 1) + c] = q.B[j0 + i + (int64_t)(c0 + c) * q.ldb];
    }
    __syncthreads();
    if (tid < nc) {
      for (int i = 0; i < b; ++i) {
        double2 s = sx[i * (TRSM_COLS + 1) + tid];
        for (int t = 0; t < i; ++t) s = cfms(D.S[t][i], sx[t * (TRSM_COLS + 1) + tid], s);
        sx[i * (TRSM_COLS + 1) + tid] = s;
      }
      if (!unit)
        for (int i = 0; i < b; ++i) sx[i * (TRSM_COLS + 1) + tid] = cmul(sx[i * (TRSM_COLS + 1) + tid], D.inv[i]);
    }
    __syncthreads();
    for (int e = tid; e < 32 * TRSM_COLS; e += TRSM_COLS) {
      const int i = e & 31, c = e >> 5;
      if (i < b && c < nc) q.B[j0 + i + (int64_t)(c0 + c) * q.ldb] = sx[(fwd ? i : b - 1 - i) * (TRSM_COLS + 1) + c];
    }
  }
}

// The update after a solved block for a few right-hand sides (nrhs <= TRSM_FEW): a thread per row,
// 64 rows a CTA, so no lane works on columns that are not there (a 32 x 32 product tile spends
// 31/32 of the FP64 pipe on them at one right-hand side).  Arguments as for k_trsm_update, whose
// order of operations it keeps.
#define TRSM_FEW 8
__global__ void __launch_bounds__(64) k_trsm_update_few(const TrsmDesc* __restrict__ d, int j0, int jb, int lower) {
  __shared__ double2 sT[32][65];
  __shared__ double2 sb[32][TRSM_FEW];
  const TrsmDesc q = d[blockIdx.y];
  if (j0 >= q.n) return;
  const int je = min(j0 + jb, q.n), kb = je - j0;
  const int m = lower ? q.n - je : j0, r0 = lower ? je : 0;
  if (m <= 0 || q.nrhs <= 0) return;
  for (int e = threadIdx.x; e < 32 * TRSM_FEW; e += 64) {
    const int t = e & 31, c = e >> 5;
    sb[t][c] = t < kb && c < q.nrhs ? q.B[j0 + t + (int64_t)c * q.ldb] : make_double2(0.0, 0.0);
  }
  for (int i0 = blockIdx.x * 64; i0 < m; i0 += gridDim.x * 64) {
    const int mm = min(64, m - i0);
    __syncthreads();
    if (q.trans) {  // op(T)[r0 + i, j0 + t] = T[j0 + t, r0 + i]: contiguous in t
      for (int e = threadIdx.x; e < 32 * 64; e += 64) {
        const int t = e & 31, i = e >> 5;
        sT[t][i] = t < kb && i < mm ? q.T[j0 + t + (int64_t)(r0 + i0 + i) * q.ldt] : make_double2(0.0, 0.0);
      }
    } else {
      const int i = threadIdx.x;
      for (int t = 0; t < 32; ++t)
        sT[t][i] = t < kb && i < mm ? q.T[r0 + i0 + i + (int64_t)(j0 + t) * q.ldt] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    if ((int)threadIdx.x < mm) {
      const int i = threadIdx.x;
#pragma unroll
      for (int c = 0; c < TRSM_FEW; ++c) {
        if (c >= q.nrhs) break;
        double2* o = q.B + r0 + i0 + i + (int64_t)c * q.ldb;
        double2 s = make_double2(0.0, 0.0);
#pragma unroll 8
        for (int t = 0; t < 32; ++t) s = cfma(sT[t][i], sb[t][c], s);
        const double2 v = *o;
        *o = make_double2(v.x - s.x, v.y - s.y);
      }
    }
  }
}

// One step for a few right-hand sides of a few matrices, a column a CTA: the update by the solved block
// [j0, j0 + jb), and the next block, solved by the CTA that has just updated its rows (tiles of 32 rows
// count from the solved block, so these are tile 0's, and stay in their registers).
// A step is a chain of FP64 instructions, and a sub-partition takes 64 clocks for each of them, whatever
// else it holds: so a lane has one real component of a row instead of a row (half the instructions a
// warp), and the two halves of the rows run on two sub-partitions, the second taking the first one's
// solutions 8 at a time.  What does not depend on B (the triangle, its reciprocals, the tile of T) is
// fetched before the wait for the step before, by programmatic launch: T is complete by then, as the
// first block's solve is an ordinary launch.  Every CTA waits, also one without work: a step's end has
// to mean that all steps before it ended.  The order of operations is that of the separate kernels.
// n = 2200, one right-hand side: 8.3 us a step (update 2.9, solve 4.2, the rest launch and exchange),
// 27 us as two launches with a row a lane.
#define TRSM_ST 64
__global__ void __launch_bounds__(TRSM_ST) k_trsm_step_few(const TrsmDesc* __restrict__ d, int j0, int jb, int lower) {
  __shared__ TrsmStage D;
  __shared__ double2 sT[32][33];
  __shared__ double sb[32][2], xs[16][2];  // re, im of the solved block; of the first half of the next
  const TrsmDesc q = d[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.z;
  const int i = 16 * warp + (lane >> 1), part = lane & 1;  // row in the order of the solve; re or im
  const int neg = part ? 0 : -1;
  auto flip = [](double v, int f) {  // -v where f: on the integer pipe
    return __hiloint2double(__double2hiint(v) ^ (f & 0x80000000), __double2loint(v));
  };
  const int je = min(j0 + jb, q.n), kb = max(0, je - j0);  // kb = 0: this matrix begins at a later block
  const int jn = lower ? j0 + jb : j0 - jb;
  const int m = kb == 0 ? 0 : lower ? q.n - je : j0;
  const bool solve = blockIdx.x == 0 && jn >= 0 && jn < q.n;
  const int b = min(jb, q.n - jn);
  const bool unit = (lower != 0) != (q.trans != 0);
  const int ntile = c < q.nrhs ? max((m + 31) / 32, solve ? 1 : 0) : 0;
  auto load_tile = [&](int tile) {  // sT[t][row of the tile, in the order of the solve]
    const int r = lower ? je + 32 * tile : j0 - 32 * tile - 1, mm = min(32, m - 32 * tile);
    double2 v[1024 / TRSM_ST];
#pragma unroll
    for (int e = 0; e < 1024 / TRSM_ST; ++e) {
      const int o = warp + e * (TRSM_ST / 32);
      const int a = q.trans ? o : lane, t = q.trans ? lane : o;  // op(T)[row a, j0 + t], contiguous in lane
      const int64_t row = lower ? r + a : r - a;
      v[e] = t < kb && a < mm ? (q.trans ? q.T[j0 + t + row * q.ldt] : q.T[row + (int64_t)(j0 + t) * q.ldt])
                              : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int e = 0; e < 1024 / TRSM_ST; ++e) {
      const int o = warp + e * (TRSM_ST / 32);
      sT[q.trans ? lane : o][q.trans ? o : lane] = v[e];
    }
  };
  if ((int)blockIdx.x < ntile) {
    load_tile(blockIdx.x);
    if (solve) trsm_stage(D, q, jn, jb, lower != 0, unit);
  }
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  double2* col = q.B + (int64_t)c * q.ldb;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    __syncthreads();
    if (tile != (int)blockIdx.x) load_tile(tile);
    const bool last = tile == 0 && solve;
    const int mm = last ? b : min(32, m - 32 * tile);
    const int row = lower ? jn + 32 * tile + i : last ? jn + b - 1 - i : j0 - 32 * tile - 1 - i;
    double x = i < mm ? __ldcg((const double*)(col + row) + part) : 0.0;
    if (kb > 0) {
      const int t = threadIdx.x >> 1;
      sb[t][part] = t < kb ? __ldcg((const double*)(col + j0 + t) + part) : 0.0;
      __syncthreads();
      double s = 0.0;
#pragma unroll 8
      for (int t = 0; t < 32; ++t) {  // cfma, one component
        const double2 v = sT[t][i];
        s = fma(v.x, sb[t][part], fma(flip(v.y, neg), sb[t][1 - part], s));
      }
      x -= s;
    }
    if (last) {
      auto take = [&](int t, double own, double other) {  // cfms, one component
        const double2 v = D.S[t][i];
        if (i > t) x = fma(-v.x, own, fma(flip(v.y, ~neg), other, x));
      };
      auto solve16 = [&](int t0, int t1) {  // rows t0 .. t1 - 1 of this warp's 16
        for (int t = t0; t < t1; ++t) {
          const int l = 2 * (t & 15);
          const double own = __shfl_sync(0xFFFFFFFFu, x, l + part), other = __shfl_sync(0xFFFFFFFFu, x, l + 1 - part);
          take(t, own, other);
        }
      };
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (warp == 0) {
          solve16(8 * h, min(b, 8 * h + 8));
          if (i >= 8 * h && i < 8 * h + 8) xs[i][part] = x;
        }
        asm volatile("bar.sync %0, 64;" ::"r"(1 + h) : "memory");
        if (warp == 1) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (8 * h + k < b) take(8 * h + k, xs[8 * h + k][part], xs[8 * h + k][1 - part]);
        }
      }
      if (warp == 1) solve16(16, b);
      if (!unit) {
        const double y = __shfl_xor_sync(0xFFFFFFFFu, x, 1);
        const double2 r = cmul(part ? make_double2(y, x) : make_double2(x, y), D.inv[i]);
        x = part ? r.y : r.x;
      }
    }
    if (i < mm) ((double*)(col + row))[part] = x;
  }
}

static cudaError_t launch_trsm_step(dim3 grid, const TrsmDesc* d, int j0, int lower, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(TRSM_ST);
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_trsm_step_few, d, j0, WSBM_NB, lower);
}

// Update after a solved diagonal block: lower: B[je:n] -= T[je:n, j0:je] B[j0:je];
// upper: B[0:j0] -= T[0:j0, j0:je] B[j0:je].
__global__ void __launch_bounds__(256) k_trsm_update(const TrsmDesc* __restrict__ d, int j0, int jb,
                                                     int lower) {
  const TrsmDesc q = d[blockIdx.y];
  if (j0 >= q.n) return;
  const int je = min(j0 + jb, q.n);
  int m = lower ? q.n - je : j0;
  if (m <= 0 || q.nrhs <= 0) return;
  int r0 = lower ? je : 0;
  int ntm = (m + GT - 1) / GT, ntn = (q.nrhs + GT - 1) / GT;
  const double2 one = make_double2(1.0, 0.0), mone = make_double2(-1.0, 0.0);
  for (int t = blockIdx.x; t < ntm * ntn; t += gridDim.x) {
    if (q.trans)  // op(T)[r0.., j0..je) = (T[j0..je, r0..])^T
      gemm_tile<true>(m, q.nrhs, je - j0, q.T + j0 + (int64_t)r0 * q.ldt, q.ldt, q.B + j0, q.ldb,
                      q.B + r0, q.ldb, mone, one, t % ntm, t / ntm);
    else
      gemm_tile<false>(m, q.nrhs, je - j0, q.T + r0 + (int64_t)j0 * q.ldt, q.ldt, q.B + j0, q.ldb,
                       q.B + r0, q.ldb, mone, one, t % ntm, t / ntm);
  }
}

// LU row interchanges on B, forward (P B) or, inverse, undone (P^T B): blocks of 256 swaps as
// gathers, one warp per column.
__global__ void __launch_bounds__(256) k_apply_piv(const TrsmDesc* __restrict__ d, int inverse) {
  __shared__ SwapLists S;
  const TrsmDesc q = d[blockIdx.y];
  if ((int)blockIdx.x * 8 >= q.nrhs) return;
  const int nblk = (q.n + 255) / 256;
  for (int k = 0; k < nblk; ++k) {
    const int j0 = (inverse ? nblk - 1 - k : k) * 256, nb = min(256, q.n - j0);
    swap_lists(S, q.piv + j0, q.n, j0, nb);
    for (int c = blockIdx.x * 8 + (threadIdx.x >> 5); c < q.nrhs; c += gridDim.x * 8)
      swap_column(S, nb, q.B + (int64_t)c * q.ldb, inverse != 0);
  }
}

// --------------------------------------------------------- fused LU + solve ----
// One CTA per matrix on a row-major working copy S of [A | B], so that a row of the trailing
// matrix is one coalesced access per warp.  Blocked right-looking LU with panels of LUS_B
// columns: the panel (rows j0..n-1) is staged in shared memory and factored by one warp with
// partial pivoting; then every thread takes one column c >= j0 + LUS_B at a time, applies the
// panel's row interchanges, solves the unit-lower L11 for its LUS_B rows of U12 and updates its
// trailing column with the rank-LUS_B product L21 U12 (one load and store per LUS_B complex
// FMAs).  Columns left of the panel only take the interchanges.  Back substitution with U on
// the B columns runs in the same blocks from the bottom, the U block column staged in shared
// memory.  Pivot choice: largest max(|re|, |im|) (integer compare of the bit patterns), first
// row on ties.
#define LUS_T 256
#define LUS_B 8

__device__ __forceinline__ unsigned long long lus_key(double2 v) {
  const unsigned long long m = 0x7fffffffffffffffull;
  const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & m;
  const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & m;
  return a > b ? a : b;
}

__device__ __forceinline__ double2* lus_col(const LuSolveDesc& q, int c) {
  return c < q.n ? q.A + (int64_t)c * q.lda : q.B + (int64_t)(c - q.n) * q.ldb;
}

// column-major [A | B] <-> row-major S through a 32 x 33 shared tile (8 warps, 4 rows each)
__device__ void lus_transpose(const LuSolveDesc& q, double2* S, int64_t ldr, double2* tile,
                              bool to_rows) {
  const int n = q.n, nc = q.n + q.nrhs;
  const int ntr = (n + 31) / 32, ntc = (nc + 31) / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int t = 0; t < ntr * ntc; ++t) {
    const int r0 = (t % ntr) * 32, c0 = (t / ntr) * 32;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int a = w + 8 * s;
      if (to_rows) {
        const int c = c0 + a, r = r0 + lane;
        if (r < n && c < nc) tile[a * 33 + lane] = lus_col(q, c)[r];
      } else {
        const int r = r0 + a, c = c0 + lane;
        if (r < n && c < nc) tile[lane * 33 + a] = S[(int64_t)r * ldr + c];
      }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int a = w + 8 * s;
      if (to_rows) {
        const int r = r0 + a, c = c0 + lane;
        if (r < n && c < nc) S[(int64_t)r * ldr + c] = tile[lane * 33 + a];
      } else {
        const int c = c0 + a, r = r0 + lane;
        if (r < n && c < nc) lus_col(q, c)[r] = tile[a * 33 + lane];
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(LUS_T) k_lu_solve_fused(const LuSolveDesc* __restrict__ d) {
  const LuSolveDesc q = d[blockIdx.x];
  const int n = q.n, nr = q.nrhs, nc = n + nr;
  if (n <= 0) return;
  const int64_t ldr = ((int64_t)nc + 7) & ~(int64_t)7;  // = wsbm_lu_solve_ldr(n, nrhs)
  double2* __restrict__ S = q.S;
  extern __shared__ double2 lus_sm[];
  double2* sinv = lus_sm;    // n pivot reciprocals
  double2* sp = lus_sm + n;  // panel / U block: LUS_B columns of stride m + 1; transpose tile
  __shared__ int spiv[LUS_B];
  const int tid = threadIdx.x, lane = tid & 31;

  lus_transpose(q, S, ldr, sp, true);
  for (int j0 = 0; j0 < n; j0 += LUS_B) {
    const int bb = min(LUS_B, n - j0), m = n - j0, ld = m + 1;
    __syncthreads();  // trailing updates of the previous panel done
    for (int e = tid; e < m * bb; e += LUS_T) {
      const int r = e / bb, t = e - r * bb;
      sp[t * ld + r] = S[(int64_t)(j0 + r) * ldr + j0 + t];
    }
    __syncthreads();
    if (tid < 32) {  // panel factorization, one warp
      for (int jj = 0; jj < bb; ++jj) {
        double2* col = sp + jj * ld;
        unsigned long long best = 0;
        int bi = 0x7fffffff;
        for (int r = jj + lane; r < m; r += 32) {
          const unsigned long long k = lus_key(col[r]);
          if (k > best || bi == 0x7fffffff) {
            best = k;
            bi = r;
          }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
          }
        }
        const int p = bi;
        if (p != jj && lane < bb) {
          double2* a = sp + lane * ld;
          const double2 x = a[jj];
          a[jj] = a[p];
          a[p] = x;
        }
        __syncwarp();
        const double2 pv = col[jj];
        const double2 inv =
            (pv.x == 0.0 && pv.y == 0.0) ? make_double2(0.0, 0.0) : cdiv(make_double2(1.0, 0.0), pv);
        if (lane == 0) {
          spiv[jj] = j0 + p;
          q.piv[j0 + jj] = j0 + p;
          sinv[j0 + jj] = inv;
        }
        for (int r = jj + 1 + lane; r < m; r += 32) col[r] = cmul(col[r], inv);
        __syncwarp();
        for (int t = jj + 1; t < bb; ++t) {
          double2* ct = sp + t * ld;
          const double2 u = ct[jj];
          for (int r = jj + 1 + lane; r < m; r += 32) ct[r] = cfms(col[r], u, ct[r]);
        }
        __syncwarp();
      }
    }
    __syncthreads();
    for (int e = tid; e < m * bb; e += LUS_T) {
      const int r = e / bb, t = e - r * bb;
      S[(int64_t)(j0 + r) * ldr + j0 + t] = sp[t * ld + r];
    }
    for (int c = tid; c < j0; c += LUS_T)  // columns of L: interchanges only
      for (int jj = 0; jj < bb; ++jj) {
        const int p = spiv[jj];
        if (p != j0 + jj) {
          double2* a = S + (int64_t)(j0 + jj) * ldr + c;
          double2* b = S + (int64_t)p * ldr + c;
          const double2 x = *a;
          *a = *b;
          *b = x;
        }
      }
    for (int c = j0 + bb + tid; c < nc; c += LUS_T) {
      double2 u[LUS_B];
#pragma unroll
      for (int jj = 0; jj < LUS_B; ++jj)
        if (jj < bb) {
          const int p = spiv[jj];
          double2* a = S + (int64_t)(j0 + jj) * ldr + c;
          if (p != j0 + jj) {
            double2* b = S + (int64_t)p * ldr + c;
            const double2 x = *a;
            *a = *b;
            *b = x;
          }
        }
#pragma unroll
      for (int t = 0; t < LUS_B; ++t)
        if (t < bb) {
          double2 v = S[(int64_t)(j0 + t) * ldr + c];
#pragma unroll
          for (int s2 = 0; s2 < t; ++s2) v = cfms(sp[s2 * ld + t], u[s2], v);
          u[t] = v;
          S[(int64_t)(j0 + t) * ldr + c] = v;
        }
      int r = bb;
      for (; r + 1 < m; r += 2) {
        double2* e0 = S + (int64_t)(j0 + r) * ldr + c;
        double2* e1 = e0 + ldr;
        double2 a0 = *e0, a1 = *e1;
#pragma unroll
        for (int t = 0; t < LUS_B; ++t)
          if (t < bb) {
            a0 = cfms(sp[t * ld + r], u[t], a0);
            a1 = cfms(sp[t * ld + r + 1], u[t], a1);
          }
        *e0 = a0;
        *e1 = a1;
      }
      if (r < m) {
        double2* e0 = S + (int64_t)(j0 + r) * ldr + c;
        double2 a0 = *e0;
#pragma unroll
        for (int t = 0; t < LUS_B; ++t)
          if (t < bb) a0 = cfms(sp[t * ld + r], u[t], a0);
        *e0 = a0;
      }
    }
  }
  // back substitution U X = Y on the B columns, block rows from the bottom
  for (int j0 = ((n - 1) / LUS_B) * LUS_B; j0 >= 0; j0 -= LUS_B) {
    const int bb = min(LUS_B, n - j0), m = j0 + bb, ld = m + 1;
    __syncthreads();
    for (int e = tid; e < m * bb; e += LUS_T) {
      const int r = e / bb, t = e - r * bb;
      sp[t * ld + r] = S[(int64_t)r * ldr + j0 + t];
    }
    __syncthreads();
    for (int c = n + tid; c < nc; c += LUS_T) {
      double2 x[LUS_B];
#pragma unroll
      for (int t = 0; t < LUS_B; ++t) x[t] = t < bb ? S[(int64_t)(j0 + t) * ldr + c] : make_double2(0.0, 0.0);
#pragma unroll
      for (int t = LUS_B - 1; t >= 0; --t)
        if (t < bb) {
          x[t] = cmul(x[t], sinv[j0 + t]);
#pragma unroll
          for (int s2 = 0; s2 < t; ++s2) x[s2] = cfms(sp[t * ld + j0 + s2], x[t], x[s2]);
        }
#pragma unroll
      for (int t = 0; t < LUS_B; ++t)
        if (t < bb) S[(int64_t)(j0 + t) * ldr + c] = x[t];
      int i = 0;
      for (; i + 1 < j0; i += 2) {
        double2* e0 = S + (int64_t)i * ldr + c;
        double2* e1 = e0 + ldr;
        double2 a0 = *e0, a1 = *e1;
#pragma unroll
        for (int t = 0; t < LUS_B; ++t)
          if (t < bb) {
            a0 = cfms(sp[t * ld + i], x[t], a0);
            a1 = cfms(sp[t * ld + i + 1], x[t], a1);
          }
        *e0 = a0;
        *e1 = a1;
      }
      if (i < j0) {
        double2* e0 = S + (int64_t)i * ldr + c;
        double2 a0 = *e0;
#pragma unroll
        for (int t = 0; t < LUS_B; ++t)
          if (t < bb) a0 = cfms(sp[t * ld + i], x[t], a0);
        *e0 = a0;
      }
    }
  }
  __syncthreads();
  lus_transpose(q, S, ldr, sp, false);
}

// ------------------------------------------------- column-pivoted Householder QR ----
// One CTA per matrix M (m x n, in place).  Step j: pivot the column of largest remaining norm
// to position j, reflect rows j..m-1 with P = I - tau u u^H (Hermitian, tau real,
// u = x - beta e1, beta = -(x0/|x0|)|x|), so P x = beta e1.  Mode 0 stops at the first j with
// |beta_j| <= tol |beta_0| (rank k = j); mode 1 runs until step kt.  The state (reflected
// matrix, exact remaining column norms, permutation) lets a later call resume.  On return
// the R factor sits in rows 0..k-1 (diagonal included; below it, reflector data).
#ifndef CPQR_CB
#define CPQR_CB 4  // default trailing columns per warp pass of the warp variant (2, 4 or 8)
#endif
#ifndef CPQR_MINB
#define CPQR_MINB 4  // minimum resident CTAs per SM asked of the register allocator (measured best)
#endif
// TPC (thread per column): each thread updates whole trailing columns against the reflector
// staged in shared memory (no warp reductions; the strided column loads stay in L1, and on
// GB300 a warp-wide DFMA takes 16 clocks, which hides them).  For matrices of up to CPQR_TPC_MAXM
// rows, the sketches: 4096 of 128 x 256 take 88 ms; from there on the two are within 4 % in large
// batches and the warps win in small ones.
#ifndef CPQR_TPC_MAXM
#define CPQR_TPC_MAXM 192
#endif
#define CPQR_CLUSTER_MAXM 12288  // rows of the cluster variant: a reflector of 192 KB in shared memory
// Warp variant: CB trailing columns per warp per pass (2*CB partial sums, a power of two <= 16).
template <bool TPC, int CB>
__global__ void __launch_bounds__(256, CPQR_MINB) k_cpqr(const QrDesc* __restrict__ d, int mode) {
  // 5 - log2(2*CB): the lane holding reduced value t is t << SH
  constexpr int SH = CB == 1 ? 4 : CB == 2 ? 3 : CB == 4 ? 2 : CB == 8 ? 1 : 0;
  extern __shared__ double2 su[];  // TPC: the reflector u = M[j:m, j]
  const QrDesc q = d[blockIdx.x];
  const int m = q.m, n = q.n;
  if (TPC ? m > CPQR_TPC_MAXM : m <= CPQR_CLUSTER_MAXM) return;
  double2* M = q.A;
  const int64_t ld = q.lda;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __shared__ double sval[256];
  __shared__ int sidx[256];
  __shared__ double s_tau;
  __shared__ double2 s_beta;
  __shared__ int s_stop;
  const int kmax = min(m, n);
  int j = q.state[0];  // resume point
  if (j == 0 && threadIdx.x == 0) q.state[1] = 0;
  // initial exact norms
  if (j == 0) {
    for (int c = warp; c < n; c += nw) {
      double s = 0.0;
      for (int i = lane; i < m; i += 32) s += cabs2(M[i + (int64_t)c * ld]);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        q.norm2[c] = s;
        q.nref[c] = s;
      }
    }
    for (int c = threadIdx.x; c < n; c += blockDim.x) q.perm[c] = c;
  }
  __syncthreads();
  const int kt = mode == 1 ? min(q.kt, kmax) : kmax;
  for (; j < kt; ++j) {
    // pivot: largest remaining norm (lowest index on ties)
    double best = -1.0;
    int bi = j;
    for (int c = j + threadIdx.x; c < n; c += blockDim.x) {
      double v = q.norm2[c];
      if (v > best) {
        best = v;
        bi = c;
      }
    }
    sval[threadIdx.x] = best;
    sidx[threadIdx.x] = bi;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        double o = sval[threadIdx.x + s];
        int oi = sidx[threadIdx.x + s];
        if (o > sval[threadIdx.x] || (o == sval[threadIdx.x] && oi < sidx[threadIdx.x])) {
          sval[threadIdx.x] = o;
          sidx[threadIdx.x] = oi;
        }
      }
      __syncthreads();
    }
    const int p = sidx[0];
    const double nrm = sqrt(fmax(sval[0], 0.0));
    if (threadIdx.x == 0) {
      int stop = 0;
      if (j == 0) q.rdiag0[0] = nrm;
      if (mode == 0 && (nrm <= q.tol * q.rdiag0[0] || nrm == 0.0)) stop = 1;
      s_stop = stop;
    }
    __syncthreads();
    if (s_stop) break;
    if (p != j) {  // swap whole columns j <-> p
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double2 t = M[i + (int64_t)j * ld];
        M[i + (int64_t)j * ld] = M[i + (int64_t)p * ld];
        M[i + (int64_t)p * ld] = t;
      }
      if (threadIdx.x == 0) {
        double t = q.norm2[j];
        q.norm2[j] = q.norm2[p];
        q.norm2[p] = t;
        t = q.nref[j];
        q.nref[j] = q.nref[p];
        q.nref[p] = t;
        int ti = q.perm[j];
        q.perm[j] = q.perm[p];
        q.perm[p] = ti;
      }
    }
    __syncthreads();
    // reflector from x = M[j:m, j]; |x| recomputed exactly
    double s = 0.0;
    for (int i = j + threadIdx.x; i < m; i += blockDim.x) s += cabs2(M[i + (int64_t)j * ld]);
    sval[threadIdx.x] = s;
    __syncthreads();
    for (int t = blockDim.x / 2; t > 0; t >>= 1) {
      if (threadIdx.x < t) sval[threadIdx.x] += sval[threadIdx.x + t];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      double xn = sqrt(sval[0]);
      double2 x0 = M[j + (int64_t)j * ld];
      double a0 = sqrt(cabs2(x0));
      double2 beta = a0 > 0.0 ? make_double2(-x0.x / a0 * xn, -x0.y / a0 * xn) : make_double2(-xn, 0.0);
      double2 u0 = make_double2(x0.x - beta.x, x0.y - beta.y);
      // u^H u = 2 |x| (|x| + |x0|)
      double uu = 2.0 * xn * (xn + a0);
      s_tau = uu > 0.0 ? 2.0 / uu : 0.0;
      s_beta = beta;
      M[j + (int64_t)j * ld] = u0;
    }
    __syncthreads();
    const double tau = s_tau;
    if (TPC) {
      const int mm = m - j;
      for (int i = threadIdx.x; i < mm; i += blockDim.x) su[i] = M[j + i + (int64_t)j * ld];
      __syncthreads();
      for (int c = j + 1 + threadIdx.x; c < n; c += blockDim.x) {
        double2* col = M + (int64_t)c * ld + j;
        double wr0 = 0.0, wi0 = 0.0, wr1 = 0.0, wi1 = 0.0;  // w = u^H col, two chains
        int i = 0;
        for (; i + 1 < mm; i += 2) {
          const double2 u0 = su[i], c0 = col[i], u1 = su[i + 1], c1 = col[i + 1];
          wr0 = fma(u0.x, c0.x, fma(u0.y, c0.y, wr0));
          wi0 = fma(u0.x, c0.y, fma(-u0.y, c0.x, wi0));
          wr1 = fma(u1.x, c1.x, fma(u1.y, c1.y, wr1));
          wi1 = fma(u1.x, c1.y, fma(-u1.y, c1.x, wi1));
        }
        if (i < mm) {
          const double2 u0 = su[i], c0 = col[i];
          wr0 = fma(u0.x, c0.x, fma(u0.y, c0.y, wr0));
          wi0 = fma(u0.x, c0.y, fma(-u0.y, c0.x, wi0));
        }
        const double2 w = make_double2(tau * (wr0 + wr1), tau * (wi0 + wi1));
        for (i = 0; i < mm; ++i) col[i] = cfms(su[i], w, col[i]);
        // remaining norm: downdate by the new row-j entry, recompute once cancellation has
        // eaten half its digits
        double nv = q.norm2[c] - cabs2(col[0]);
        if (nv <= 1e-8 * q.nref[c]) {
          double ns = 0.0;
          for (i = 1; i < mm; ++i) ns += cabs2(col[i]);
          nv = ns;
          q.nref[c] = ns;
        }
        q.norm2[c] = fmax(nv, 0.0);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        q.tauv[j] = tau;
        q.betav[j] = s_beta;
      }
      __syncthreads();
      continue;
    }
    // apply P to the trailing columns: a warp takes CB columns at a time, so each element
    // of u is loaded once for all of them and the 2*CB partial dot products are summed
    // across the warp by recursive halving (each level hands half of the values to the partner
    // lane; 2*CB - 1 + (5 - log2(2*CB)) adds per lane instead of 10 per column).  The remaining
    // norm is downdated by the new row-j entry and recomputed exactly once cancellation has
    // eaten half its digits (remaining norm below 1e-8 of the last exact one).
    const double2* u = M + (int64_t)j * ld;
    for (int c0 = j + 1 + warp * CB; c0 < n; c0 += nw * CB) {
      const int nc = min(CB, n - c0);
      double acc[2 * CB];  // re of the nc columns, then im
#pragma unroll
      for (int v = 0; v < 2 * CB; ++v) acc[v] = 0.0;
      for (int i = j + lane; i < m; i += 32) {  // w = u^H col, as fused multiply-adds
        const double2 ui = u[i];
#pragma unroll
        for (int v = 0; v < CB; ++v) {
          if (v < nc) {
            const double2 ci = M[i + (int64_t)(c0 + v) * ld];
            acc[v] = fma(ui.x, ci.x, fma(ui.y, ci.y, acc[v]));
            acc[CB + v] = fma(ui.x, ci.y, fma(-ui.y, ci.x, acc[CB + v]));
          }
        }
      }
      int cur = 2 * CB;
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        if (cur > 1) {
          const int h = cur >> 1;
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int v = 0; v < CB; ++v) {
            if (v < h) {
              const double send = up ? acc[v] : acc[v + h];
              const double keep = up ? acc[v + h] : acc[v];
              acc[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          cur = h;
        } else {
          acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
        }
      }
      // value t (re of column t for t < CB, im of column t - CB otherwise) sits in lane t << SH
      double2 w[CB];
#pragma unroll
      for (int v = 0; v < CB; ++v) {
        w[v].x = tau * __shfl_sync(0xffffffffu, acc[0], v << SH);
        w[v].y = tau * __shfl_sync(0xffffffffu, acc[0], (CB + v) << SH);
      }
      for (int i = j + lane; i < m; i += 32) {
        const double2 ui = u[i];
#pragma unroll
        for (int v = 0; v < CB; ++v) {
          if (v < nc) {
            double2* pc = M + i + (int64_t)(c0 + v) * ld;
            *pc = cfms(ui, w[v], *pc);
          }
        }
      }
      __syncwarp();
      for (int v = 0; v < nc; ++v) {
        const int c = c0 + v;
        const double2* col = M + (int64_t)c * ld;
        const double rj = cabs2(col[j]);  // the new row-j entry (written by lane 0)
        double nv = q.norm2[c] - rj;
        if (nv <= 1e-8 * q.nref[c]) {
          double ns = 0.0;
          for (int i = j + 1 + lane; i < m; i += 32) ns += cabs2(col[i]);
          for (int o = 16; o > 0; o >>= 1) ns += __shfl_xor_sync(0xffffffffu, ns, o);
          nv = ns;
          __syncwarp();
          if (lane == 0) q.nref[c] = ns;
        }
        __syncwarp();
        if (lane == 0) q.norm2[c] = fmax(nv, 0.0);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      q.tauv[j] = tau;
      q.betav[j] = s_beta;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    q.state[0] = j;
    q.state[1] = j;  // rank reached
  }
}

// One matrix of more than CPQR_TPC_MAXM and at most CPQR_CLUSTER_MAXM rows per cluster of 1 to 8 CTAs: more than one where there
// are too few matrices to fill the GPU (the upper tree levels: few boxes, the largest matrices).
// The trailing columns are dealt to the warps of the whole cluster, CB at a time; a column's sums
// do not depend on which warp or how many CTAs take it, so a matrix has the same factor in every
// batch.  Every CTA finds the pivot from the norms in
// global memory by itself and stages the pivot column as the reflector in its own shared memory,
// so a step costs two cluster barriers: one between that staging and the update (which overwrites
// the pivot's slot with column j), one after the update (the ID of the 16384-node star, 64 to 256
// matrices a level: 257 -> 88 ms).  The reflectors are not kept (only R and
// the trailing matrix are read later): column j's rows below j stay as they are.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void cpqr_sync(uint32_t csize) {
  if (csize == 1)
    __syncthreads();
  else
    cluster_sync_all();
}

// Norms in an order that integers have: negative zero and NaN never win.
__device__ __forceinline__ long long cpqr_norm_key(double v) {
  const long long b = __double_as_longlong(v);
  return (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll ? -1 : b;
}

template <int CB, int MINB>
__global__ void __launch_bounds__(256, MINB) k_cpqr_cluster(const QrDesc* __restrict__ d, int mode) {
  constexpr int SH = CB == 1 ? 4 : CB == 2 ? 3 : CB == 4 ? 2 : 1;  // 5 - log2(2 * CB)
  extern __shared__ double2 su[];  // the reflector u = (column p)[j : m]
  uint32_t rank, csize;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
  const QrDesc q = d[blockIdx.x / csize];
  const int m = q.m, n = q.n;
  if (m <= CPQR_TPC_MAXM || m > CPQR_CLUSTER_MAXM) return;  // another kernel's
  double2* M = q.A;
  const int64_t ld = q.lda;
  const int tid = threadIdx.x, lane = tid & 31, nw = blockDim.x >> 5;
  const int gw = (int)rank * nw + (tid >> 5), gn = (int)csize * nw;  // this warp and all warps of the cluster
  __shared__ long long sval[8];
  __shared__ double ssum[8];
  __shared__ int sidx[8], s_stop;
  __shared__ double s_tau;
  __shared__ double2 s_beta;
  const int kmax = min(m, n);
  int j = q.state[0];  // resume point
  if (j == 0) {
    for (int c = gw; c < n; c += gn) {
      double s = 0.0;
      for (int i = lane; i < m; i += 32) s += cabs2(M[i + (int64_t)c * ld]);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        q.norm2[c] = s;
        q.nref[c] = s;
        q.perm[c] = c;
      }
    }
  }
  cpqr_sync(csize);
  const int kt = mode == 1 ? min(q.kt, kmax) : kmax;
  for (; j < kt; ++j) {
    // pivot: largest remaining norm (lowest index on ties), compared by bits on the integer pipe: an
    // FP64 instruction of a warp takes its sub-partition 64 clocks, a compare too
    long long best = -1;
    int p = j;
    for (int c = j + tid; c < n; c += blockDim.x) {
      const long long v = cpqr_norm_key(__ldcg(q.norm2 + c));
      if (v > best) {
        best = v;
        p = c;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, p, o);
      if (ob > best || (ob == best && oi < p)) {
        best = ob;
        p = oi;
      }
    }
    if (lane == 0) {
      sval[tid >> 5] = best;
      sidx[tid >> 5] = p;
    }
    __syncthreads();
    best = sval[0];
    p = sidx[0];
    for (int w = 1; w < nw; ++w)
      if (sval[w] > best || (sval[w] == best && sidx[w] < p)) {
        best = sval[w];
        p = sidx[w];
      }
    // reflector from x = column p; |x| recomputed exactly
    const int mm = m - j;
    double s = 0.0;
    for (int i = tid; i < mm; i += blockDim.x) {
      const double2 v = __ldcg(M + j + i + (int64_t)p * ld);
      su[i] = v;
      s += cabs2(v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ssum[tid >> 5] = s;
    __syncthreads();
    // the scalars, a lane for each root and each quotient: one root and one quotient long
    if (tid < 32) {
      double t = lane < nw ? ssum[lane] : 0.0;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      const double2 x0 = su[0];
      const double rt = sqrt(lane == 1 ? cabs2(x0) : t);
      const double xn = __shfl_sync(0xffffffffu, rt, 0), a0 = __shfl_sync(0xffffffffu, rt, 1);
      const double uu = 2.0 * xn * (xn + a0);  // u^H u = 2 |x| (|x| + |x0|)
      const double qt = (lane == 0 ? -x0.x : lane == 1 ? -x0.y : 2.0) / (lane < 2 ? a0 : uu);
      const double bx = __shfl_sync(0xffffffffu, qt, 0), by = __shfl_sync(0xffffffffu, qt, 1);
      const double tq = __shfl_sync(0xffffffffu, qt, 2);
      if (lane == 0) {
        const double2 beta = a0 > 0.0 ? make_double2(bx * xn, by * xn) : make_double2(-xn, 0.0);
        su[0] = make_double2(x0.x - beta.x, x0.y - beta.y);
        s_tau = uu > 0.0 ? tq : 0.0;
        s_beta = beta;
      }
    } else if (tid == 32) {  // beside them, the stopping rule: the same in every CTA
      const double nrm = sqrt(best > 0 ? __longlong_as_double(best) : 0.0);
      if (j == 0 && rank == 0) q.rdiag0[0] = nrm;
      const double r00 = j == 0 ? nrm : __ldcg(q.rdiag0);
      s_stop = mode == 0 && (nrm <= q.tol * r00 || nrm == 0.0);
    }
    cpqr_sync(csize);
    if (s_stop) break;
    const double tau = s_tau;
    if (rank == 0 && tid == 0) {
      q.tauv[j] = tau;
      q.betav[j] = s_beta;
      if (p != j) {
        const int t = q.perm[j];
        q.perm[j] = q.perm[p];
        q.perm[p] = t;
      }
    }
    // P applied to the trailing columns; slot p takes column j (the interchange)
    for (int c0 = j + 1 + gw * CB; c0 < n; c0 += gn * CB) {
      const int nc = min(CB, n - c0);
      const double2* src[CB];
#pragma unroll
      for (int v = 0; v < CB; ++v) src[v] = M + j + (int64_t)(c0 + v == p ? j : (v < nc ? c0 + v : c0)) * ld;
      double acc[2 * CB];  // re of the CB columns, then im
#pragma unroll
      for (int v = 0; v < 2 * CB; ++v) acc[v] = 0.0;
      for (int i = lane; i < mm; i += 32) {
        const double2 ui = su[i];
#pragma unroll
        for (int v = 0; v < CB; ++v) {
          const double2 ci = src[v][i];
          acc[v] = fma(ui.x, ci.x, fma(ui.y, ci.y, acc[v]));
          acc[CB + v] = fma(ui.x, ci.y, fma(-ui.y, ci.x, acc[CB + v]));
        }
      }
      int cur = 2 * CB;
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        if (cur > 1) {
          const int h = cur >> 1;
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int v = 0; v < CB; ++v) {
            if (v < h) {
              const double send = up ? acc[v] : acc[v + h];
              const double keep = up ? acc[v + h] : acc[v];
              acc[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          cur = h;
        } else {
          acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
        }
      }
      acc[0] *= tau;
      double2 w[CB], top[CB];
#pragma unroll
      for (int v = 0; v < CB; ++v) {
        w[v].x = __shfl_sync(0xffffffffu, acc[0], v << SH);
        w[v].y = __shfl_sync(0xffffffffu, acc[0], (CB + v) << SH);
        top[v] = make_double2(0.0, 0.0);
      }
      for (int i = lane; i < mm; i += 32) {
        const double2 ui = su[i];
#pragma unroll
        for (int v = 0; v < CB; ++v)
          if (v < nc) {
            const double2 x = cfms(ui, w[v], src[v][i]);
            M[j + i + (int64_t)(c0 + v) * ld] = x;
            if (i == 0) top[v] = x;
          }
      }
      // remaining norms: downdated by the new row-j entry, recomputed exactly once cancellation
      // has eaten half their digits; column v's in lane v
      double2 mine = make_double2(0.0, 0.0);
#pragma unroll
      for (int v = 0; v < CB; ++v) {
        const double tx = __shfl_sync(0xffffffffu, top[v].x, 0), ty = __shfl_sync(0xffffffffu, top[v].y, 0);
        if (lane == v) mine = make_double2(tx, ty);
      }
      const bool on = lane < nc;
      const int lc = c0 + lane, ls = lc == p ? j : lc;
      const double nf = on ? __ldcg(q.nref + ls) : 0.0;
      double nv = (on ? __ldcg(q.norm2 + ls) : 1.0) - cabs2(mine);
      const unsigned redo = __ballot_sync(0xffffffffu, on && nv <= 1e-8 * nf);
      if (redo) __syncwarp();  // a vote does not order memory: the sums below read other lanes' stores
#pragma unroll
      for (int v = 0; v < CB; ++v)
        if (redo >> v & 1) {
          double ns = 0.0;
          const double2* col = M + (int64_t)(c0 + v) * ld;
          for (int i = j + 1 + lane; i < m; i += 32) ns += cabs2(col[i]);
          for (int o = 16; o > 0; o >>= 1) ns += __shfl_xor_sync(0xffffffffu, ns, o);
          if (lane == v) {
            nv = ns;
            q.nref[lc] = ns;
          }
        }
      if (on) {
        if (ls != lc && !(redo >> lane & 1)) q.nref[lc] = nf;
        q.norm2[lc] = fmax(nv, 0.0);
      }
      if (c0 <= p && p < c0 + nc)  // rows above j of R: plain interchange of columns j and p
        for (int i = lane; i < j; i += 32) {
          const double2 t = M[i + (int64_t)j * ld];
          M[i + (int64_t)j * ld] = M[i + (int64_t)p * ld];
          M[i + (int64_t)p * ld] = t;
        }
    }
    cpqr_sync(csize);
  }
  if (rank == 0 && tid == 0) {
    q.state[0] = j;
    q.state[1] = j;  // rank reached
  }
}

// After the QR: put the diagonal of R back (the reflectors are no longer needed) and zero
// the part of column t below the diagonal within the first k rows (none: R11 is k x k).
__global__ void k_cpqr_finish(const QrDesc* __restrict__ d) {
  const QrDesc q = d[blockIdx.x];
  int k = q.state[1];
  for (int t = threadIdx.x; t < k; t += blockDim.x) q.A[t + (int64_t)t * q.lda] = q.betav[t];
}

// ------------------------------------------------------------------ host drivers ----
static int grid_cap() { return wsbm_sm_count() * 8; }

static int tiles_x(int64_t tiles) {
  int cap = grid_cap();
  return (int)(tiles < 1 ? 1 : (tiles < cap ? tiles : cap));
}

// The batched kernels below index their descriptor by blockIdx.y; a batch of more than
// LAUNCH_MAX_Y matrices runs as consecutive chunks (the matrices are independent).
#define LAUNCH_MAX_Y 65535

int wsbm_gemm_batched(const GemmDesc* d_desc, int nbatch, int max_m, int max_n, cudaStream_t st) {
  if (nbatch <= 0) return 0;
  if (nbatch > LAUNCH_MAX_Y) {
    for (int c = 0; c < nbatch; c += LAUNCH_MAX_Y)
      if (int rc = wsbm_gemm_batched(d_desc + c, std::min(LAUNCH_MAX_Y, nbatch - c), max_m, max_n, st))
        return rc;
    return 0;
  }
  if (max_n <= 0) return 0;
  // few columns: a 32 x 32 tile would leave 3/4 of its lanes (8 columns) to 31/32 (one) without work
  // (one column of the box solves at N = 4096: 162 us a launch as tiles, 18 us here)
  if (max_n <= GEMM_FEW) {
    k_gemm_few<<<dim3(tiles_x((max_m + 63) / 64), nbatch, max_n), 128, 0, st>>>(d_desc);
  } else {
    int64_t t = (int64_t)((max_m + GT - 1) / GT) * ((max_n + GT - 1) / GT);
    dim3 grid(tiles_x(t), nbatch);
    k_gemm<<<grid, 256, 0, st>>>(d_desc, nbatch);
  }
  wsbm_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int wsbm_lu_batched(const LuDesc* d_desc, int nbatch, int max_n, int* d_info, cudaStream_t st) {
  if (nbatch <= 0) return 0;
  if (nbatch > LAUNCH_MAX_Y) {
    for (int c = 0; c < nbatch; c += LAUNCH_MAX_Y)
      if (int rc = wsbm_lu_batched(d_desc + c, std::min(LAUNCH_MAX_Y, nbatch - c), max_n,
                                   d_info ? d_info + c : nullptr, st))
        return rc;
    return 0;
  }
  for (int j0 = 0; j0 < max_n; j0 += WSBM_NB) {
    k_lu_panel<<<nbatch, 256, 0, st>>>(d_desc, j0, WSBM_NB, d_info);
    wsbm_count_launch();
    dim3 gs(tiles_x((max_n + 127) / 128), nbatch);
    k_laswp<<<gs, 128, 0, st>>>(d_desc, j0, WSBM_NB);
    wsbm_count_launch();
    k_lu_trsm_row<<<gs, 128, 0, st>>>(d_desc, j0, WSBM_NB);
    wsbm_count_launch();
    int m = max_n - j0 - WSBM_NB;
    if (m > 0) {
      int64_t t = (int64_t)((m + GT - 1) / GT) * ((m + GT - 1) / GT);
      dim3 gg(tiles_x(t), nbatch);
      k_lu_update<<<gg, 256, 0, st>>>(d_desc, j0, WSBM_NB);
      wsbm_count_launch();
    }
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// Triangular solves T^-1 B (lower unit: forward; upper non-unit: backward), blocked.
int wsbm_trsm_batched(const TrsmDesc* d_desc, int nbatch, int max_n, int max_nrhs, int lower,
                      cudaStream_t st) {
  if (nbatch <= 0 || max_n <= 0 || max_nrhs <= 0) return 0;
  if (nbatch > LAUNCH_MAX_Y) {
    for (int c = 0; c < nbatch; c += LAUNCH_MAX_Y)
      if (int rc = wsbm_trsm_batched(d_desc + c, std::min(LAUNCH_MAX_Y, nbatch - c), max_n, max_nrhs,
                                     lower, st))
        return rc;
    return 0;
  }
  // blocks of WSBM_NB rows: the diagonal block, then the update of the rows still to solve.  One
  // warp per column while the columns are few (measured equal at about 4000 on 152 SMs)
  const bool warps = (int64_t)nbatch * max_nrhs <= (int64_t)wsbm_sm_count() * 24;
  const size_t smx = (size_t)32 * (TRSM_COLS + 1) * sizeof(double2);
  if (!warps && wsbm_smem_optin((const void*)k_trsm_diag, 64 * 1024) != cudaSuccess) return -3;
  const int nblk = (max_n + WSBM_NB - 1) / WSBM_NB;
  const bool few = max_nrhs <= TRSM_FEW, steps = warps && few;
  for (int k = 0; k < nblk; ++k) {
    const int j0 = (lower ? k : nblk - 1 - k) * WSBM_NB;
    if (k == 0 || !steps) {  // a step solves the block after it
      if (warps)
        k_trsm_diag_warp<<<dim3(tiles_x((max_nrhs + 3) / 4), nbatch), 128, 0, st>>>(d_desc, j0, WSBM_NB, lower);
      else
        k_trsm_diag<<<dim3(tiles_x((max_nrhs + TRSM_COLS - 1) / TRSM_COLS), nbatch), TRSM_COLS, smx, st>>>(
            d_desc, j0, WSBM_NB, lower);
      wsbm_count_launch();
    }
    const int m = lower ? max_n - j0 - WSBM_NB : j0;
    if (m <= 0) continue;
    if (steps) {
      if (launch_trsm_step(dim3(tiles_x((m + 31) / 32), nbatch, max_nrhs), d_desc, j0, lower, st) != cudaSuccess) return -3;
    } else if (few) {
      k_trsm_update_few<<<dim3(tiles_x((m + 63) / 64), nbatch), 64, 0, st>>>(d_desc, j0, WSBM_NB, lower);
    } else {
      const int64_t t = (int64_t)((m + GT - 1) / GT) * ((max_nrhs + GT - 1) / GT);
      k_trsm_update<<<dim3(tiles_x(t), nbatch), 256, 0, st>>>(d_desc, j0, WSBM_NB, lower);
    }
    wsbm_count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// Upper-triangular backward solves must start at each matrix's own last block; the blocked
// loop above runs from the batch maximum, and blocks with j0 >= n skip, so a smaller matrix
// simply starts later.  (Each k_trsm_diag / k_trsm_update guards j0 >= n.)

int wsbm_lu_solve_batched(const TrsmDesc* d_desc_lower, const TrsmDesc* d_desc_upper, int nbatch,
                          int max_n, int max_nrhs, cudaStream_t st) {
  if (nbatch <= 0) return 0;
  if (nbatch > LAUNCH_MAX_Y) {
    for (int c = 0; c < nbatch; c += LAUNCH_MAX_Y)
      if (int rc = wsbm_lu_solve_batched(d_desc_lower + c, d_desc_upper + c,
                                         std::min(LAUNCH_MAX_Y, nbatch - c), max_n, max_nrhs, st))
        return rc;
    return 0;
  }
  k_apply_piv<<<dim3(tiles_x((max_nrhs + 7) / 8), nbatch), 256, 0, st>>>(d_desc_lower, 0);
  wsbm_count_launch();
  int rc = wsbm_trsm_batched(d_desc_lower, nbatch, max_n, max_nrhs, 1, st);
  if (rc) return rc;
  return wsbm_trsm_batched(d_desc_upper, nbatch, max_n, max_nrhs, 0, st);
}

int64_t wsbm_lu_solve_ldr(int n, int nrhs) { return ((int64_t)n + nrhs + 7) & ~(int64_t)7; }

int wsbm_lu_solve_fused_batched(const LuSolveDesc* d_desc, int nbatch, int max_n, int max_nc,
                                cudaStream_t st) {
  if (nbatch <= 0) return 0;
  if (max_n > WSBM_LUS_MAXN || max_n > max_nc) return -1;
  const size_t tile = 32 * 33, panel = (size_t)(max_n + 1) * LUS_B;
  const size_t sm = ((size_t)max_n + (panel > tile ? panel : tile)) * sizeof(double2);
  // the opt-in above 48 KB is a per-device attribute of the kernel
  if (wsbm_smem_optin((const void*)k_lu_solve_fused, sm) != cudaSuccess) return -3;
  k_lu_solve_fused<<<nbatch, LUS_T, sm, st>>>(d_desc);
  wsbm_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int wsbm_cpqr_tpc_rows() { return CPQR_TPC_MAXM; }

template <int CB, int MINB>
static int launch_cpqr_cluster(const QrDesc* d_desc, int nbatch, int mode, int cl, int max_m, cudaStream_t st) {
  const size_t sm = (size_t)std::min(max_m, CPQR_CLUSTER_MAXM) * sizeof(double2);
  if (wsbm_smem_optin((const void*)k_cpqr_cluster<CB, MINB>, sm) != cudaSuccess) return -3;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(nbatch * cl));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  wsbm_count_launch();
  return cudaLaunchKernelEx(&cfg, k_cpqr_cluster<CB, MINB>, d_desc, mode) == cudaSuccess ? 0 : -3;
}

// The kernel is chosen per matrix, by its rows, so that its factor does not depend on the others of
// the launch: each launch skips the matrices of the other kinds.
int wsbm_cpqr_batched(const QrDesc* d_desc, int nbatch, int nsmall, int mode, int max_m, cudaStream_t st) {
  if (nbatch <= 0) return 0;
  const WsbmTune tu = wsbm_tune_current();
  if (nsmall > 0) {
    const int thr = tu.cpqr_threads == 128 ? 128 : 256;
    k_cpqr<true, CPQR_CB><<<nbatch, thr, (size_t)std::min(max_m, CPQR_TPC_MAXM) * sizeof(double2), st>>>(d_desc, mode);
    wsbm_count_launch();
  }
  const int nbig = nbatch - nsmall;
  if (nbig > 0) {
    // 2, 4 or 8 CTAs per matrix while the GPU holds them all at once (three per SM)
    int cl = 1;
    while (cl < 8 && (int64_t)nbig * cl * 2 <= (int64_t)wsbm_sm_count() * 3) cl *= 2;
    // columns a warp takes at a time (its sums are the same): 4 share the reductions of short columns, 2 give
    // a matrix alone more warps (4096 of 256 x 256: 204 ms with 4, 231 with 2, 196 in the thread-per-column
    // kernel; 1200 of 400 x 300: 136, 144, 137; one of 500 x 400: 8.2, 5.8, 49)
    const int cb = max_m <= 2048 ? 2 : tu.cpqr_cb;
    if (int rc = cl == 1 && max_m <= 800 ? launch_cpqr_cluster<4, 3>(d_desc, nbatch, mode, cl, max_m, st)
                 : cb == 2               ? launch_cpqr_cluster<2, 3>(d_desc, nbatch, mode, cl, max_m, st)
                 : cb == 8               ? launch_cpqr_cluster<8, 2>(d_desc, nbatch, mode, cl, max_m, st)
                                         : launch_cpqr_cluster<4, 2>(d_desc, nbatch, mode, cl, max_m, st))
      return rc;
  }
  if (max_m > CPQR_CLUSTER_MAXM) {
    k_cpqr<false, 4><<<nbatch, 256, 0, st>>>(d_desc, mode);
    wsbm_count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int wsbm_cpqr_finish(const QrDesc* d_desc, int nbatch, cudaStream_t st) {
  if (nbatch <= 0) return 0;
  k_cpqr_finish<<<nbatch, 128, 0, st>>>(d_desc);
  wsbm_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int wsbm_lu_solve_t_batched(const TrsmDesc* d_desc, int nbatch, int max_n, int max_nrhs,
                            cudaStream_t st) {
  if (nbatch <= 0) return 0;
  if (nbatch > LAUNCH_MAX_Y) {
    for (int c = 0; c < nbatch; c += LAUNCH_MAX_Y)
      if (int rc = wsbm_lu_solve_t_batched(d_desc + c, std::min(LAUNCH_MAX_Y, nbatch - c), max_n,
                                           max_nrhs, st))
        return rc;
    return 0;
  }
  int rc = wsbm_trsm_batched(d_desc, nbatch, max_n, max_nrhs, 1, st);  // U^T, forward
  if (rc) return rc;
  rc = wsbm_trsm_batched(d_desc, nbatch, max_n, max_nrhs, 0, st);  // L^T, backward
  if (rc) return rc;
  k_apply_piv<<<dim3(tiles_x((max_nrhs + 7) / 8), nbatch), 256, 0, st>>>(d_desc, 1);
  wsbm_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ----------------------------------------------- batched LU + solve on the tensor cores ----
// The box factors of a level (LU(D) with D^-1 L, and Dhat = M^-1) as a blocked right-looking LU
// with LUT_NB-column panels over every box of the batch at once: per panel, the panel is
// factored with partial pivoting on the FP64 pipe (k_lu_panel, one CTA per matrix), its row
// swaps are applied to the rest of A and to B, U12 = L11^-1 A12 (and L11^-1 B12) and the
// trailing update A22 -= L21 U12 (B22 likewise) run as batched products on the tensor cores
// (wsbm_zgemm_tc_batched, two items per box: the A part and the B part), with L11^-1 formed
// explicitly per box.  The back substitution X = U^-1 B runs by panels from the bottom:
// X_p = U_pp^-1 X_p and X_{<p} -= U_{<p,p} X_p, again as batched tensor-core products.
// Same factors (L unit lower, U, piv[j] = the row swapped with row j) and solution as
// k_lu_solve_fused, to rounding; pivoting by |a|^2 (k_lu_panel).
#define LUT_NB 64

// Apply the swaps piv[j0 .. je) to the columns of A outside [j0, je) and to every column of B.
__global__ void k_lut_swap(const LuSolveDesc* __restrict__ d, int j0, int jb) {
  const LuSolveDesc q = d[blockIdx.y];
  if (j0 >= q.n) return;
  const int je = min(j0 + jb, q.n), nc = q.n + q.nrhs;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    if (c >= j0 && c < je) continue;
    double2* col = c < q.n ? q.A + (int64_t)c * q.lda : q.B + (int64_t)(c - q.n) * q.ldb;
    for (int j = j0; j < je; ++j) {
      const int p = q.piv[j];
      if (p != j) {
        const double2 t = col[j];
        col[j] = col[p];
        col[p] = t;
      }
    }
  }
}

// X = inverse of the unit lower (upper = 0) or of the upper (upper = 1, non-unit) triangle of
// the diagonal block A[j0 : j0+jb, j0 : j0+jb] (jb <= 64) of item blockIdx.y; X: jb x jb (ld jb) at
// X + blockIdx.y * ldx_item.  One warp per column, 16 columns a CTA.
__global__ void __launch_bounds__(512) k_lut_trinv(const LuSolveDesc* __restrict__ d, int j0, int jb, int upper,
                                                   double2* __restrict__ Xall, int64_t ldx_item) {
  __shared__ double2 stage[32 * 64];
  __shared__ double2 dinv[32];
  const LuSolveDesc q = d[blockIdx.y];
  if (j0 >= q.n) return;
  const int b = min(jb, q.n - j0), j = blockIdx.x * 16 + (threadIdx.x >> 5);
  if ((int)blockIdx.x * 16 >= b) return;
  double2* x = Xall + blockIdx.y * ldx_item + (int64_t)j * b;
  const double2* T = q.A + j0 + (int64_t)j0 * q.lda;
  const int first = blockIdx.x / 2;  // 16 columns a CTA lie in one slot of 32
  if (upper)
    tri_inverse_column<2, true>(T, q.lda, b, j, x, stage, dinv, true, first);
  else
    tri_inverse_column<2, false>(T, q.lda, b, j, x, stage, dinv, true, first);
}

// Inverses of the diagonal blocks of LU factors (unit lower L, upper U), for block triangular
// solves whose products run on the tensor cores.  Item blockIdx.y with block width nb = q.nb,
// block p = blockIdx.x / NCH (rows and columns p nb .. min(n, (p + 1) nb)), blockIdx.z = 0: L_pp^-1
// into Linv + p nb^2, 1: U_pp^-1 into Uinv + p nb^2 (column-major, leading dimension nb; the
// part outside a ragged last block is not written).  One warp per column, 16 columns a CTA (chunk
// blockIdx.x % NCH).  A zero diagonal entry of U leaves a zero row in U_pp^-1.
#define DINV_CHUNKS 16  // CTAs per block: up to 256 columns
__global__ void __launch_bounds__(512) k_lu_dinv(const DinvDesc* __restrict__ d) {
  extern __shared__ double2 stage[];
  __shared__ double2 dinv[32];
  const DinvDesc q = d[blockIdx.y];
  const int nb = q.nb, p = blockIdx.x / DINV_CHUNKS, ch = blockIdx.x % DINV_CHUNKS, j0 = p * nb;
  if (j0 >= q.n) return;
  const int b = min(nb, q.n - j0), j = ch * 16 + (threadIdx.x >> 5);
  if (ch * 16 >= b) return;
  const bool upper = blockIdx.z != 0;
  double2* x = (upper ? q.Uinv : q.Linv) + (int64_t)p * nb * nb + (int64_t)j * nb;
  const double2* T = q.A + j0 + (int64_t)j0 * q.lda;
  if (upper)
    tri_inverse_column<8, true>(T, q.lda, b, j, x, stage, dinv, true, ch / 2);
  else
    tri_inverse_column<8, false>(T, q.lda, b, j, x, stage, dinv, true, ch / 2);
}

int wsbm_lu_dinv_batched(const DinvDesc* d_desc, int nitems, int max_blocks, int max_nb, cudaStream_t st) {
  if (nitems <= 0 || max_blocks <= 0) return 0;
  if (max_nb < 1 || max_nb > 256) return -1;
  const size_t sm = (size_t)32 * 256 * sizeof(double2);
  if (wsbm_smem_optin((const void*)k_lu_dinv, sm) != cudaSuccess) return -3;
  for (int c = 0; c < nitems; c += LAUNCH_MAX_Y) {
    const int n = std::min(LAUNCH_MAX_Y, nitems - c);
    k_lu_dinv<<<dim3(max_blocks * DINV_CHUNKS, n, 2), 512, sm, st>>>(d_desc + c);
    wsbm_count_launch();
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// perm of the row interchanges piv (piv[j]: the row swapped with row j at step j, j = 0..n-1):
// (P b)[r] = b[perm[r]].  One CTA per item, 256 swaps at a time.
__global__ void __launch_bounds__(256) k_piv_perm(const PermDesc* __restrict__ d) {
  __shared__ SwapLists S;
  const PermDesc q = d[blockIdx.x];
  const int t = threadIdx.x;
  for (int r = t; r < q.n; r += 256) q.perm[r] = r;
  for (int j0 = 0; j0 < q.n; j0 += 256) {
    const int nb = min(256, q.n - j0);
    swap_lists(S, q.piv + j0, q.n, j0, nb);
    int v[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = t + 256 * h;
      if (e < 2 * nb && S.dst[e] >= 0) v[h] = q.perm[S.src[e]];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = t + 256 * h;
      if (e < 2 * nb && S.dst[e] >= 0) q.perm[S.dst[e]] = v[h];
    }
  }
}

int wsbm_piv_perm_batched(const PermDesc* d_desc, int nitems, cudaStream_t st) {
  if (nitems <= 0) return 0;
  k_piv_perm<<<nitems, 256, 0, st>>>(d_desc);
  wsbm_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

size_t wsbm_lu_solve_tc_ws_bytes(const LuSolveDesc* h, int nbatch) {
  // the largest product step: two items per box (A part and B part) of the first panel
  std::vector<TcProduct> p;
  p.reserve(2 * (size_t)nbatch);
  int maxn = 0;
  for (int i = 0; i < nbatch; ++i) {
    TcProduct a;
    memset(&a, 0, sizeof(a));
    a.m = h[i].n;
    a.n = h[i].n;
    a.k = LUT_NB;
    p.push_back(a);
    a.n = h[i].nrhs > 0 ? h[i].nrhs : 1;
    p.push_back(a);
    maxn = std::max(maxn, h[i].n);
  }
  size_t b = wsbm_zgemm_tc_batched_ws_bytes(p.data(), (int)p.size());
  b = (b + 255) & ~(size_t)255;
  b += (size_t)nbatch * LUT_NB * LUT_NB * sizeof(double2) + 256;  // diagonal-block inverses
  return b;
}

int wsbm_lu_solve_tc_batched(const LuSolveDesc* h, const LuSolveDesc* d, int nbatch, const LuDesc* d_lu,
                             void* ws, cudaStream_t st) {
  return wsbm_lu_solve_tc_batched_nb(h, d, nbatch, d_lu, ws, st, wsbm_tune_current().box_nb);
}

int wsbm_lu_solve_tc_batched_nb(const LuSolveDesc* h, const LuSolveDesc* d, int nbatch, const LuDesc* d_lu,
                                void* ws, cudaStream_t st, int nb) {
  if (nbatch <= 0) return 0;
  if (nb < 8 || nb > LUT_NB || nb % 8) return -1;
  if (nbatch > 32767 || !h || !d || !d_lu || !ws) return -1;
  int maxn = 0, maxnc = 0;
  for (int i = 0; i < nbatch; ++i) {
    maxn = std::max(maxn, h[i].n);
    maxnc = std::max(maxnc, h[i].n + h[i].nrhs);
  }
  size_t off = wsbm_zgemm_tc_ws_bytes(1, 1, 1);  // recomputed below for the actual products
  {
    std::vector<TcProduct> p(2 * (size_t)nbatch);
    for (int i = 0; i < nbatch; ++i) {
      memset(&p[2 * i], 0, 2 * sizeof(TcProduct));
      p[2 * i].m = p[2 * i + 1].m = h[i].n;
      p[2 * i].n = h[i].n;
      p[2 * i + 1].n = h[i].nrhs > 0 ? h[i].nrhs : 1;
      p[2 * i].k = p[2 * i + 1].k = LUT_NB;
    }
    off = (wsbm_zgemm_tc_batched_ws_bytes(p.data(), (int)p.size()) + 255) & ~(size_t)255;
  }
  double2* X = (double2*)((char*)ws + off);  // LUT_NB x LUT_NB per box
  const int64_t ldx = (int64_t)LUT_NB * LUT_NB;
  const double2 one = make_double2(1.0, 0.0), mone = make_double2(-1.0, 0.0), zero = make_double2(0.0, 0.0);
  std::vector<TcProduct> items;
  items.reserve(2 * (size_t)nbatch);
  auto run = [&](double2 alpha, double2 beta) -> int {
    if (items.empty()) return 0;
    int rc = wsbm_zgemm_tc_batched(items.data(), (int)items.size(), alpha, beta, ws, st);
    items.clear();
    return rc;
  };
  auto add = [&](const double2* A, int64_t lda, const double2* B, int64_t ldb, double2* C, int64_t ldc, int m,
                 int n, int k) {
    if (m <= 0 || n <= 0 || k <= 0) return;
    TcProduct t;
    t.A = A;
    t.lda = lda;
    t.B = B;
    t.ldb = ldb;
    t.C = C;
    t.ldc = ldc;
    t.m = m;
    t.n = n;
    t.k = k;
    t.pad = 0;
    items.push_back(t);
  };
  // ---- factorization
  for (int j0 = 0; j0 < maxn; j0 += nb) {
    k_lu_panel<<<nbatch, 256, 0, st>>>(d_lu, j0, nb, nullptr);
    k_lut_swap<<<dim3(tiles_x((maxnc + 127) / 128), nbatch), 128, 0, st>>>(d, j0, nb);
    k_lut_trinv<<<dim3((nb + 15) / 16, nbatch), 512, 0, st>>>(d, j0, nb, 0, X, ldx);
    wsbm_count_launches(3);
    // U12 = L11^-1 [A12 | B1]  (in place: the digit planes are formed before C is written)
    for (int i = 0; i < nbatch; ++i) {
      const LuSolveDesc& q = h[i];
      if (j0 >= q.n) continue;
      const int jb = std::min(nb, q.n - j0), je = j0 + jb;
      const double2* Li = X + i * ldx;
      add(Li, jb, q.A + j0 + (int64_t)je * q.lda, q.lda, q.A + j0 + (int64_t)je * q.lda, q.lda, jb, q.n - je, jb);
      add(Li, jb, q.B + j0, q.ldb, q.B + j0, q.ldb, jb, q.nrhs, jb);
    }
    if (int rc = run(one, zero)) return rc;
    // A22 -= L21 U12, B2 -= L21 U12_B
    for (int i = 0; i < nbatch; ++i) {
      const LuSolveDesc& q = h[i];
      if (j0 >= q.n) continue;
      const int jb = std::min(nb, q.n - j0), je = j0 + jb;
      const double2* L21 = q.A + je + (int64_t)j0 * q.lda;
      add(L21, q.lda, q.A + j0 + (int64_t)je * q.lda, q.lda, q.A + je + (int64_t)je * q.lda, q.lda, q.n - je,
          q.n - je, jb);
      add(L21, q.lda, q.B + j0, q.ldb, q.B + je, q.ldb, q.n - je, q.nrhs, jb);
    }
    if (int rc = run(mone, one)) return rc;
  }
  // ---- back substitution X = U^-1 (L^-1 P B), panels from the bottom
  for (int j0 = ((maxn - 1) / nb) * nb; j0 >= 0; j0 -= nb) {
    k_lut_trinv<<<dim3((nb + 15) / 16, nbatch), 512, 0, st>>>(d, j0, nb, 1, X, ldx);
    wsbm_count_launch();
    for (int i = 0; i < nbatch; ++i) {
      const LuSolveDesc& q = h[i];
      if (j0 >= q.n) continue;
      const int jb = std::min(nb, q.n - j0);
      add(X + i * ldx, jb, q.B + j0, q.ldb, q.B + j0, q.ldb, jb, q.nrhs, jb);
    }
    if (int rc = run(one, zero)) return rc;
    for (int i = 0; i < nbatch; ++i) {
      const LuSolveDesc& q = h[i];
      if (j0 >= q.n || j0 == 0) continue;
      const int jb = std::min(nb, q.n - j0);
      add(q.A + (int64_t)j0 * q.lda, q.lda, q.B + j0, q.ldb, q.B, q.ldb, j0, q.nrhs, jb);
    }
    if (int rc = run(mone, one)) return rc;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}
