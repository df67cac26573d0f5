// LU with partial pivoting of large complex matrices (the dense roots of a build): one, or the roots of
// several curves in step, panel by panel in the same launches.  Every kernel works on a matrix without regard
// to the others, so the factors of a root do not depend on its company.
//
// Right-looking, outer panels of LUB_NB columns (LUB_NB_BIG for large n, where the deeper
// tensor-core products pay for the longer panels).  An outer panel is factored recursively by
// halves down to base panels of at most 32 columns; a base panel is one cooperative launch over
// the whole GPU (k_lub_panel).  The updates between the halves, U12 = L11^-1 A12 and the
// trailing update A22 -= L21 U12 run on the tensor cores (wsbm_zgemm_tc).  Factors and piv as
// for wsbm_lu_batched.  Pivot: the row of largest max(|re|, |im|) compared on the upper 32 bits
// of its bit pattern (within 2^-20 of the largest), first row on ties.
#include <algorithm>
#include <climits>
#include <vector>

#include "cplx.cuh"
#include "dense.h"
#include "rowswap.cuh"
#include "tri.cuh"

#ifndef LUB_NB
#define LUB_NB 128      // outer panel width
#endif
#ifndef LUB_NB_BIG
#define LUB_NB_BIG 256  // outer panel width from LUB_BIG_N on: deeper tensor-core products
#endif
#ifndef LUB_BIG_N
// 256 columns from here on only: at n = 8200 they take 95 ms against 107, but their wider explicit
// inverses cost accuracy (random matrix, rms of PA - LU over |A|: 4.4e-14 against 2.7e-14; 2.75e-14 with
// the launch-per-column version).  n = 12288: 200 ms against 245, n = 16384: 368 against 489.
#define LUB_BIG_N 12288
#endif
#define LUB_W 32            // widest base panel: one lane per column
#define LUB_T 256           // threads of a base-panel CTA
#define LUB_MINROWS 32      // fewest rows per CTA (the base panel's pivot rows all start in CTA 0)
#define LUB_MAXCTA 256      // CTAs a base panel can use (key slots per column)
#define LUB_MAXB 16         // matrices in step (their descriptors are kernel arguments)
#define LUB_SMEM (200 * 1024)
#define LUB_WAIT_NS 2000000000ull  // bound of every wait (2 s)

static __device__ int g_lub_error;  // set when a bounded wait ran out

struct LubItem {
  double2* A;
  int64_t lda;
  int n;
  int *piv, *info;
  unsigned long long* slots;  // [outer panel's columns][LUB_MAXCTA]
  double2 *cand, *diag, *inv;
};
struct LubBatch {
  LubItem it[LUB_MAXB];     // by falling n
  int first[LUB_MAXB + 1];  // base panel: first CTA of each
  int R;                    // base panel: rows per CTA
};

__device__ __forceinline__ unsigned long long lub_key(double2 v, int row) {
  const unsigned long long m = 0x7fffffffffffffffull;
  const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & m;
  const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & m;
  const unsigned long long hi = (a > b ? a : b) >> 32;
  return (hi << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)row);
}

// by 32-bit reductions of the halves: about 80 clocks, a tree of 64-bit shuffles 400, four times a column
__device__ __forceinline__ unsigned long long lub_warp_max(unsigned long long best) {
  const unsigned hi = (unsigned)(best >> 32), mh = __reduce_max_sync(0xFFFFFFFFu, hi);
  const unsigned ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? (unsigned)best : 0u);
  return (unsigned long long)mh << 32 | ml;
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long lub_time() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Base panel: columns [c0, min(c1, n)) (at most 32) of rows [c0, n), rows spread over the CTAs of one
// cooperative launch, R consecutive rows each (R >= w), held in shared memory from the first to
// the last column.  Several matrices share the launch, each with CTAs of its own that wait for one another only.  Per column every CTA publishes its best candidate (key) and that candidate's
// panel row; every CTA then reads all the keys, takes the winner's row as the pivot row and
// updates its own rows, so a column costs one exchange through L2 instead of two launches.  Bound by
// that exchange (release, 152 polled keys, one row read): 3.8 us a column at n = 8200, 31 ms in all.
// Only the next column is updated before its candidate is published, the others while it travels (with
// the whole update first, and 64-bit reductions, 6.4 us; launches per column and their gaps 100 ms).
// The others take the pivots two at a time, j even and j + 1, their products summed before the one
// subtraction: an entry is rounded at its own size once a pair (a multiply-add per product would round it
// four times).  1/2 on the diagonal, rms of PA - LU there in ulp(1/2): n = 2048 0.91, 8200 1.68 (a pivot at a
// time 1.43, 2.08; 8-column panels with products between them 0.89, 1.63).
//   slots  key slots [w][LUB_MAXCTA], zero on entry (a key is never zero)
//   cand   published rows [2][LUB_MAXCTA][32]; a slot of one parity is rewritten two columns
//          later, after every CTA has published the column between (and so has read it)
//   diag   row c as its owner holds it before the swap, [2][32]
__global__ void __launch_bounds__(LUB_T, 1)
    k_lub_panel(const __grid_constant__ LubBatch q, int c0, int c1, int slot0) {
  extern __shared__ double2 sm[];
  int it = 0;
  while ((int)blockIdx.x >= q.first[it + 1]) ++it;
  double2* __restrict__ A = q.it[it].A;
  const int64_t lda = q.it[it].lda;
  const int n = q.it[it].n, w = min(c1, n) - c0, R = q.R;
  unsigned long long* slots = q.it[it].slots + (size_t)slot0 * LUB_MAXCTA;
  double2 *cand = q.it[it].cand, *diag = q.it[it].diag;
  int *__restrict__ piv = q.it[it].piv, *__restrict__ info = q.it[it].info;
  const int RS = R | 1;  // odd stride: a row read across the columns meets no bank twice
  __shared__ double2 prow[4][LUB_W];  // rows of the last four pivots, by column modulo 4
  __shared__ double2 s_inv;
  __shared__ unsigned long long red[LUB_T / 32], keys[LUB_T / 32];
  __shared__ int s_err;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = (int)blockIdx.x - q.first[it], G = q.first[it + 1] - q.first[it];
  const int r0 = c0 + b * R, cnt = min(R, n - r0);
  for (int e = tid; e < R * w; e += LUB_T) {
    const int t = e / R, i = e - t * R;
    if (i < cnt) sm[t * RS + i] = A[(int64_t)(r0 + i) + (int64_t)(c0 + t) * lda];
  }
  if (tid == 0) s_err = 0;
  __syncthreads();
  unsigned long long best = 0;
  for (int i = tid; i < cnt; i += LUB_T) {
    const unsigned long long k = lub_key(sm[i], r0 + i);
    best = k > best ? k : best;
  }
  int prev = 0;  // first row below the last pivot's: rows from here on await its update
  // a lane per real component where a step waits for the result: half the FP64 instructions a warp
  const int part = lane & 1;
  auto flip = [part](double v) {  // -v for the real part: on the integer pipe
    return __hiloint2double(__double2hiint(v) ^ (part ? 0 : (int)0x80000000), __double2loint(v));
  };
  auto comp = [part](const double2& v, int other) { return (part ^ other) ? v.y : v.x; };
  auto dot = [&](double x, const double2& l, const double2& u) {  // x plus the product's component
    return fma(l.x, comp(u, 0), fma(flip(l.y), comp(u, 1), x));
  };

  for (int j = 0; j < w; ++j) {
    const int c = c0 + j;
    best = lub_warp_max(best);
    if (lane == 0) red[warp] = best;
    __syncthreads();
    unsigned long long* row = slots + (size_t)j * LUB_MAXCTA;
    // Column j is up to date.  At an even j the columns after it await the pivots j - 2 and j - 1: those
    // before `half` take them now, the others at j + 1, when all await pivot j as well.
    const int je = j & ~1, half = je + 1 + max(2, (w - je) / 2);
    const bool pair = je > 0, odd = j & 1;
    const double2 *ra = prow[(je - 2) & 3], *rb = prow[(je - 1) & 3], *rc = prow[je & 3];
    // The candidate's row (warps 0 and 1) is published complete, but for the columns from `half` on at an odd
    // j; row c (warps 2 and 3 of its CTA) as the rows in shared memory will be after this update.
    unsigned long long k = 0;
    if (warp < (b == 0 ? 4 : 2)) {
      k = lub_warp_max(lane < LUB_T / 32 ? red[lane] : 0ull);
      const bool mine = warp < 2;
      const int loc = mine ? (int)(0xFFFFFFFFu - (unsigned)k) - r0 : j, t = 16 * (warp & 1) + (lane >> 1);
      if (t < w) {
        double x = comp(sm[t * RS + loc], 0);
        if (t > j) {
          if (mine && odd) {
            if (t < half) x -= dot(0.0, sm[je * RS + loc], rc[t]);
          } else if (pair && (mine || (t >= half) == odd)) {
            x -= dot(dot(0.0, sm[(je - 1) * RS + loc], rb[t]), sm[(je - 2) * RS + loc], ra[t]);
          }
        }
        double2* o = mine ? cand + ((size_t)(j & 1) * LUB_MAXCTA + b) * LUB_W : diag + (j & 1) * LUB_W;
        __stcg((double*)(o + t) + part, x);
      }
    }
    __syncthreads();
    if (tid == 0) st_release(row + b, k);
    if (pair) {  // while the candidates travel
      const int t0 = odd ? half : j + 1, t1 = odd ? w : min(half, w), rows = cnt - prev;
      for (int e = tid; e < rows * (t1 - t0); e += LUB_T) {  // (row, column) packed: no lane without a row
        const int q = e / rows, i = prev + e - q * rows, t = t0 + q;
        const double2 v = cfma(sm[(je - 2) * RS + i], ra[t], cmul(sm[(je - 1) * RS + i], rb[t])), x = sm[t * RS + i];
        sm[t * RS + i] = make_double2(x.x - v.x, x.y - v.y);
      }
    }
    // all keys of this column, a thread each (bounded); a warp that read several in turn would wait
    // for L2 several times
    unsigned long long top = 0;
    if (tid < G) {
      top = ld_acquire(row + tid);
      if (top == 0) {
        const unsigned long long t0 = lub_time();
        for (unsigned it = 1; (top = ld_acquire(row + tid)) == 0; ++it) {
          if ((it & 63) == 0 && (*(volatile int*)&g_lub_error || lub_time() - t0 > LUB_WAIT_NS)) {
            atomicExch(&g_lub_error, 1);
            s_err = 1;
            break;
          }
        }
      }
    }
    top = lub_warp_max(top);
    if (lane == 0) keys[warp] = top;
    __syncthreads();
    if (s_err) return;
    if (warp == 0) {
      top = lub_warp_max(lane < LUB_T / 32 ? keys[lane] : 0ull);
      const int p = (int)(0xFFFFFFFFu - (unsigned)top), bp = (p - c0) / R;
      if (lane < w) {
        const double2 v = __ldcg(cand + ((size_t)(j & 1) * LUB_MAXCTA + bp) * LUB_W + lane);
        prow[j & 3][lane] = v;
        if (p != c && b == bp) sm[lane * RS + (p - r0)] = __ldcg(diag + (j & 1) * LUB_W + lane);
        if (b == 0) sm[lane * RS + j] = v;
        if (lane == j) {
          const bool zero = v.x == 0.0 && v.y == 0.0;
          s_inv = zero ? make_double2(0.0, 0.0) : cdiv(make_double2(1.0, 0.0), v);
          if (b == 0) {
            piv[c] = p;
            if (zero && info) info[0] = c + 1;
          }
        }
      }
    }
    __syncthreads();
    // rows below c: multipliers, and the next column with its candidate; the rest follows the publication
    const int first = b == 0 ? j + 1 : 0;
    const double2 iv = s_inv;
    best = 0;
    for (int i0 = first; i0 < cnt; i0 += LUB_T / 2) {  // the same for every lane
      const int i = i0 + (tid >> 1), ii = min(i, cnt - 1);
      const double2 a = sm[j * RS + ii];
      const double l = fma(comp(a, 0), iv.x, flip(comp(a, 1) * iv.y)), lo = __shfl_xor_sync(0xFFFFFFFFu, l, 1);
      __syncwarp();
      if (i < cnt) ((double*)&sm[j * RS + i])[part] = l;
      if (j + 1 < w) {
        const double2 u1 = prow[j & 3][j + 1];
        double s = fma(part ? lo : l, comp(u1, 0), flip((part ? l : lo) * comp(u1, 1)));
        if (odd) s = dot(s, sm[je * RS + ii], rc[j + 1]);
        const double v = comp(sm[(j + 1) * RS + ii], 0) - s;
        const int h = __double2hiint(v) & 0x7fffffff, ho = __shfl_xor_sync(0xFFFFFFFFu, h, 1);
        if (i < cnt) {
          ((double*)&sm[(j + 1) * RS + i])[part] = v;
          const unsigned long long x = (unsigned long long)max(h, ho) << 32 | (0xFFFFFFFFu - (unsigned)(r0 + i));
          best = x > best ? x : best;
        }
      }
    }
    // an odd j's pivot row from `half` on (at most 15 columns), by the last warp, a lane per component
    const int t = half + (lane >> 1);
    if (warp == LUB_T / 32 - 1 && odd && t < w) {
      double2* r = prow[j & 3];
      double x = comp(r[t], 0);
      if (pair) x -= dot(dot(0.0, r[je - 1], rb[t]), r[je - 2], ra[t]);
      x -= dot(0.0, r[je], rc[t]);
      ((double*)&r[t])[part] = x;
      if (b == 0) ((double*)&sm[t * RS + j])[part] = x;
    }
    prev = first;
  }
  __syncthreads();
  for (int e = tid; e < R * w; e += LUB_T) {
    const int t = e / R, i = e - t * R;
    if (i < cnt) A[(int64_t)(r0 + i) + (int64_t)(c0 + t) * lda] = sm[t * RS + i];
  }
}

// Row interchanges piv[j0 .. min(j0 + nb, n)) (nb <= 256) on the columns [a0, a1) and [b0, min(b1, n)), as
// one gather per column, one warp each: the top nb rows are read and written contiguously (5 us a
// call at n = 8200).  Matrix blockIdx.y.
__global__ void __launch_bounds__(256)
    k_lub_rowswap(const __grid_constant__ LubBatch q, int j0, int nb, int a0, int a1, int b0, int b1) {
  __shared__ SwapLists S;
  const LubItem& x = q.it[blockIdx.y];
  const int jb = min(nb, x.n - j0), na = a1 - a0, tot = na + max(0, min(b1, x.n) - b0);
  if ((int)blockIdx.x * 8 >= tot) return;
  swap_lists(S, x.piv + j0, x.n, j0, jb);
  for (int c = blockIdx.x * 8 + (threadIdx.x >> 5); c < tot; c += gridDim.x * 8)
    swap_column(S, jb, x.A + (int64_t)(c < na ? a0 + c : b0 + (c - na)) * x.lda, false);
}

// X = L^-1 B for the unit lower triangle L of A[r0 : r0 + nb, r0 : r0 + nb] (nb <= 32 NS), one warp
// per column (tri.cuh), `cols` columns a CTA (the other warps help to stage L: the solves are bound
// by FP64, so one column per SM until there are more columns than SMs).  B: the columns [b0, min(b1, n)) of A's
// rows r0 .. r0 + nb - 1, in place; b0 < 0: the inverse itself, into `inv` (leading dimension nb).  Matrix
// blockIdx.y.
template <int NS>
__global__ void __launch_bounds__(128)
    k_lub_trsm(const __grid_constant__ LubBatch p, int r0, int nb, int b0, int b1, int cols) {
  extern __shared__ double2 stage[];
  const LubItem& m = p.it[blockIdx.y];
  const int ncols = b0 < 0 ? nb : min(b1, m.n) - b0;
  if ((int)blockIdx.x * cols >= ncols) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = blockIdx.x * cols + warp;
  const bool on = warp < cols && q < ncols;
  const double2* L = m.A + r0 + (int64_t)r0 * m.lda;
  if (b0 < 0) {
    tri_inverse_column<NS, false>(L, m.lda, nb, q, m.inv + (int64_t)q * nb, stage, nullptr, on, (int)blockIdx.x * cols / 32);
    return;
  }
  double2 x[NS];
  double2* col = m.A + r0 + (int64_t)(b0 + q) * m.lda;
#pragma unroll
  for (int s = 0; s < NS; ++s)
    x[s] = on && s * 32 + lane < nb ? col[s * 32 + lane] : make_double2(0.0, 0.0);
  tri_solve_warp<NS, false>(L, m.lda, nb, x, stage, nullptr, on);
#pragma unroll
  for (int s = 0; s < NS; ++s)
    if (on && s * 32 + lane < nb) col[s * 32 + lane] = x[s];
}

namespace {
// Matrices in step.  Panels are those of the largest; a smaller one leaves with the panel that reaches its
// last column, whose part beyond it is empty.
struct Lub {
  LubBatch q;
  int count, nb, base;
  cudaStream_t st;
  int cs;                       // first column of the outer panel
  void* ws;                     // work space of the tensor-core products
  size_t wsb;                   // and its size
  std::vector<TcProduct> prod;  // the products of one step

  int n(int i) const { return q.it[i].n; }
  int beyond(int c) const {  // matrices of more than c columns
    int k = 0;
    while (k < count && n(k) > c) ++k;
    return k;
  }

  int panel(int c0, int c1) {
    const int k = beyond(c0), nsm = std::min(wsbm_sm_count(), LUB_MAXCTA);
    int64_t rows = 0;
    for (int i = 0; i < k; ++i) rows += n(i) - c0;
    int R = (int)std::max<int64_t>(LUB_MINROWS, (rows + nsm - 1) / nsm);
    for (;; ++R) {
      q.first[0] = 0;
      for (int i = 0; i < k; ++i) q.first[i + 1] = q.first[i] + (n(i) - c0 + R - 1) / R;
      if (q.first[k] <= nsm) break;
    }
    q.R = R;
    const size_t smem = (size_t)(c1 - c0) * (R | 1) * sizeof(double2);
    if (smem > LUB_SMEM || wsbm_smem_optin((const void*)k_lub_panel, LUB_SMEM) != cudaSuccess) return -3;
    int slot0 = c0 - cs;
    void* args[] = {&q, &c0, &c1, &slot0};
    if (cudaLaunchCooperativeKernel((const void*)k_lub_panel, dim3(q.first[k]), dim3(LUB_T), args, smem, st) != cudaSuccess)
      return -3;
    wsbm_count_launch();
    return 0;
  }

  void swap(int j0, int w, int a0, int a1, int b0, int b1) {
    const int k = beyond(j0), tot = (a1 - a0) + std::max(0, std::min(b1, n(0)) - b0);
    if (tot <= 0) return;
    const int cap = std::max(1, wsbm_sm_count() * 4 / k);
    k_lub_rowswap<<<dim3(std::min((tot + 7) / 8, cap), k), 256, 0, st>>>(q, j0, w, a0, a1, b0, b1);
    wsbm_count_launch();
  }

  template <int NS>
  int trsm_ns(int r0, int w, int b0, int b1, int k) {
    const size_t sm = (size_t)32 * 32 * NS * sizeof(double2);
    if (wsbm_smem_optin((const void*)k_lub_trsm<NS>, sm) != cudaSuccess) return -3;
    const int ncols = b0 < 0 ? w : std::min(b1, n(0)) - b0;
    const int cols = std::min(4, (ncols * k + wsbm_sm_count() - 1) / wsbm_sm_count());
    k_lub_trsm<NS><<<dim3((ncols + cols - 1) / cols, k), 128, sm, st>>>(q, r0, w, b0, b1, cols);
    wsbm_count_launch();
    return 0;
  }
  int trsm(int r0, int w, int b0, int b1, int k) {  // on the first k matrices
    if (w <= 32) return trsm_ns<1>(r0, w, b0, b1, k);
    if (w <= 64) return trsm_ns<2>(r0, w, b0, b1, k);
    if (w <= 128) return trsm_ns<4>(r0, w, b0, b1, k);
    return trsm_ns<8>(r0, w, b0, b1, k);
  }

  void add(const double2* A, int64_t lda, const double2* B, int64_t ldb, double2* C, int64_t ldc, int m, int nn, int k) {
    if (m > 0 && nn > 0) prod.push_back({A, lda, B, ldb, C, ldc, m, nn, k, 0});
  }
  int run(double alpha, double beta) {
    int rc = 0;
    const double2 a = make_double2(alpha, 0.0), b = make_double2(beta, 0.0);
    if (prod.size() == 1) {
      const TcProduct& t = prod[0];
      rc = wsbm_zgemm_tc(t.m, t.n, t.k, a, t.A, t.lda, t.B, t.ldb, b, t.C, t.ldc, ws, wsb, st);
    } else if (!prod.empty()) {
      rc = wsbm_zgemm_tc_batched(prod.data(), (int)prod.size(), a, b, ws, st);
    }
    prod.clear();
    return rc;
  }

  // factor columns [c0, c1) of rows [c0, n); row swaps across the whole outer panel
  int rec(int c0, int c1) {
    if (beyond(c0) == 0) return 0;
    if (c1 - c0 <= base) {
      if (int rc = panel(c0, c1)) return rc;
      swap(c0, c1 - c0, cs, c0, c1, cs + nb);
      return 0;
    }
    const int mid = c0 + (c1 - c0) / 2, k = beyond(mid);
    if (int rc = rec(c0, mid)) return rc;
    if (k == 0) return 0;
    // A[c0:mid, mid:c1] = L11^-1 A[c0:mid, mid:c1];  A[mid:n, mid:c1] -= A[mid:n, c0:mid] A[c0:mid, mid:c1]
    if (int rc = trsm(c0, mid - c0, mid, c1, k)) return rc;
    for (int i = 0; i < k; ++i) {
      const LubItem& x = q.it[i];
      add(x.A + mid + (int64_t)c0 * x.lda, x.lda, x.A + c0 + (int64_t)mid * x.lda, x.lda,
          x.A + mid + (int64_t)mid * x.lda, x.lda, x.n - mid, std::min(c1, x.n) - mid, mid - c0);
    }
    if (int rc = run(-1.0, 1.0)) return rc;
    return rec(mid, c1);
  }

  int factor() {
    for (int j0 = 0; j0 < n(0); j0 += nb) {
      const int je = j0 + nb, k = beyond(je);
      cs = j0;
      if (cudaMemsetAsync(q.it[0].slots, 0, (size_t)beyond(j0) * nb * LUB_MAXCTA * sizeof(unsigned long long), st) !=
          cudaSuccess)
        return -3;
      if (int rc = rec(j0, je)) return rc;
      swap(j0, nb, 0, j0, je, INT_MAX);
      if (k == 0) continue;
      // U12 = L11^-1 A12 as a tensor-core product with the explicit inverse of the unit lower
      // L11 (the digit planes of A12 are formed before A12 is overwritten)
      if (int rc = trsm(j0, nb, -1, 0, k)) return rc;
      for (int i = 0; i < k; ++i) {
        const LubItem& x = q.it[i];
        double2* U = x.A + j0 + (int64_t)je * x.lda;
        add(x.inv, nb, U, x.lda, U, x.lda, nb, x.n - je, nb);
      }
      if (int rc = run(1.0, 0.0)) return rc;
      for (int i = 0; i < k; ++i) {
        const LubItem& x = q.it[i];
        add(x.A + je + (int64_t)j0 * x.lda, x.lda, x.A + j0 + (int64_t)je * x.lda, x.lda,
            x.A + je + (int64_t)je * x.lda, x.lda, x.n - je, x.n - je, nb);
      }
      if (int rc = run(-1.0, 1.0)) return rc;
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
  }
};

// columns a base panel can take: every CTA holds its rows of them in shared memory
int lub_base_width(int n) {
  const int64_t per = std::max<int64_t>(LUB_MINROWS, (n + wsbm_sm_count() - 1) / wsbm_sm_count()) + 1;
  for (int w = LUB_W; w > 1; w /= 2)
    if (per * w * (int64_t)sizeof(double2) <= LUB_SMEM) return w;
  return 1;
}

// work space: the products' planes, then key slots, published rows and L11^-1 of each matrix
constexpr size_t lub_slot_bytes = (size_t)LUB_NB_BIG * LUB_MAXCTA * sizeof(unsigned long long);
constexpr size_t lub_cand_bytes = (size_t)2 * (LUB_MAXCTA + 1) * LUB_W * sizeof(double2);
constexpr size_t lub_inv_bytes = (size_t)LUB_NB_BIG * LUB_NB_BIG * sizeof(double2);
size_t lub_product_bytes(const LuDesc* h, int count) {
  size_t b = wsbm_zgemm_tc_ws_bytes(h[0].n, h[0].n, LUB_NB_BIG);  // either panel width fits
  if (count > 1) {
    std::vector<TcProduct> p(count);
    for (int i = 0; i < count; ++i) p[i] = {nullptr, 0, nullptr, 0, nullptr, 0, h[i].n, h[i].n, LUB_NB, 0};
    b = std::max(b, wsbm_zgemm_tc_batched_ws_bytes(p.data(), count));
  }
  return (b + 255) & ~(size_t)255;
}

int lub_run(const LuDesc* h, int count, int* d_info, void* ws, cudaStream_t st, int nb) {
  Lub x;
  x.count = count;
  x.nb = nb;
  x.base = std::min(lub_base_width(h[0].n), nb);
  x.st = st;
  x.ws = ws;
  x.wsb = lub_product_bytes(h, count);
  char* slots = (char*)ws + x.wsb;
  char* cand = slots + count * lub_slot_bytes;
  char* inv = cand + count * lub_cand_bytes;
  for (int i = 0; i < count; ++i) {
    double2* c = (double2*)(cand + i * lub_cand_bytes);
    x.q.it[i] = {h[i].A, h[i].lda, h[i].n, h[i].piv, d_info,
                 (unsigned long long*)slots + (size_t)i * nb * LUB_MAXCTA,  // without a gap: one memset
                 c, c + (size_t)2 * LUB_MAXCTA * LUB_W, (double2*)(inv + i * lub_inv_bytes)};
  }
  return x.factor();
}
}  // namespace

int wsbm_lu_big_large_n() { return LUB_BIG_N; }

// outer panel width: the tuned one of n's size class (LUB_NB / LUB_NB_BIG by default)
static int lub_nb(int n) {
  const WsbmTune t = wsbm_tune_current();
  return n >= LUB_BIG_N ? t.root_nb_large : t.root_nb_mid;
}

size_t wsbm_lu_big_multi_ws_bytes(const LuDesc* h, int count) {
  if (count <= 0 || h[0].n <= 0) return 256;
  return lub_product_bytes(h, count) + count * (lub_slot_bytes + lub_cand_bytes + lub_inv_bytes) + 256;
}

size_t wsbm_lu_big_ws_bytes(int n) {
  const LuDesc d = {nullptr, n, nullptr, n, 0};
  return wsbm_lu_big_multi_ws_bytes(&d, 1);
}

int wsbm_lu_big_multi_max(const LuDesc* h, int count) {
  if (lub_nb(h[0].n) != LUB_NB) return 1;  // wide panels are worth their launches alone
  const int nsm = std::min(wsbm_sm_count(), LUB_MAXCTA);
  int64_t rows = 0;
  int k = 0;
  // rows a CTA has to hold of 32 columns when every matrix rounds up to whole CTAs
  for (; k < std::min(count, LUB_MAXB); ++k) {
    rows += h[k].n;
    if (lub_nb(h[k].n) != LUB_NB) break;
    if (k > 0 && (nsm <= k + 1 || ((rows + nsm - k - 2) / (nsm - k - 1) + 1) * LUB_W * (int64_t)sizeof(double2) > LUB_SMEM))
      break;
  }
  return std::max(k, 1);
}

int wsbm_lu_big_multi(const LuDesc* h, int count, void* ws, cudaStream_t st) {
  if (count <= 0) return 0;
  if (!h || !ws || ((uintptr_t)ws & 255) || count > wsbm_lu_big_multi_max(h, count)) return -1;
  for (int i = 0; i < count; ++i)
    if (!h[i].A || !h[i].piv || h[i].n <= 0 || h[i].lda < h[i].n || (i && h[i].n > h[i - 1].n)) return -1;
  return lub_run(h, count, nullptr, ws, st, lub_nb(h[0].n));
}

int wsbm_lu_big(double2* A, int64_t lda, int n, int* piv, int* d_info, void* ws, cudaStream_t st) {
  return wsbm_lu_big_nb(A, lda, n, piv, d_info, ws, st, lub_nb(n));
}

int wsbm_lu_big_nb(double2* A, int64_t lda, int n, int* piv, int* d_info, void* ws, cudaStream_t st, int nb) {
  if (n <= 0) return 0;
  if (!A || !piv || !ws || lda < n || ((uintptr_t)ws & 255)) return -1;
  if (nb != LUB_NB && nb != LUB_NB_BIG) return -1;
  const LuDesc d = {A, lda, piv, n, 0};
  return lub_run(&d, 1, d_info, ws, st, nb);
}

// Error flags of the bounded waits of the panel and of its products: reads and clears both
// (synchronizes the stream).
int wsbm_lu_big_status(cudaStream_t st, int n) {
  const int rc = wsbm_zgemm_tc_status(st, n > 512);  // smaller results never come from residues
  if (rc == -3) return rc;
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_lub_error, sizeof(int)) != cudaSuccess) return -3;
  if (v) {
    const int z = 0;
    cudaMemcpyToSymbol(g_lub_error, &z, sizeof(int));
    return -5;
  }
  return rc;
}
