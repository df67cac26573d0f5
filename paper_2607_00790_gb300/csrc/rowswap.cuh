// Row interchanges of an LU as gathers.
#pragma once
#include <cuda_runtime.h>

// Shared memory of swap_lists.
struct SwapLists {
  int sp[256], ptr[256], src[512], dst[512];
};

// The interchanges "row j0 + t with row piv[t]", t = 0 .. nb - 1 in that order (nb <= 256, piv in
// global memory), as at most 2 nb moves: row S.dst[e] receives the content of row S.src[e],
// e < 2 nb, none where S.dst[e] < 0.  With a[t] the row whose content sits in row j0 + t just
// before swap t, row j0 + t ends with the content of row piv[t] and a row below the block with
// the content a[t] of the last swap that names it.  Entries of piv outside [j0 + t, n) count as
// no swap.  Called by a CTA of 256 threads; ends with a barrier.
__device__ __forceinline__ void swap_lists(SwapLists& S, const int* __restrict__ piv, int n, int j0, int nb) {
  const int t = threadIdx.x;
  __syncthreads();  // an earlier list is done with
  if (t < nb) {
    const int p = piv[t];
    S.sp[t] = p >= j0 + t && p < n ? p : j0 + t;
  }
  __syncthreads();
  int par = -1, prev = -1;
  bool last = true;
  if (t < nb) {
    for (int i = 0; i < nb; ++i) {
      const int q = S.sp[i];
      if (i < t && q == j0 + t) par = i;
      if (i < t && q == S.sp[t]) prev = i;
      if (i > t && q == S.sp[t]) last = false;
    }
    S.ptr[t] = par >= 0 ? par : t;
  }
  __syncthreads();
  for (int s = 1; s < nb; s <<= 1) {  // root of each chain by pointer jumping
    const int v = t < nb ? S.ptr[S.ptr[t]] : 0;
    __syncthreads();
    if (t < nb) S.ptr[t] = v;
    __syncthreads();
  }
  if (t < nb) {
    const int at = j0 + S.ptr[t];
    S.dst[t] = j0 + t;
    S.src[t] = S.sp[t] == j0 + t ? at : (prev >= 0 ? j0 + S.ptr[prev] : S.sp[t]);
    S.dst[nb + t] = S.sp[t] >= j0 + nb && last ? S.sp[t] : -1;
    S.src[nb + t] = at;
  }
  __syncthreads();
}

// The moves on one column, by one warp; `inverse` undoes them.
__device__ __forceinline__ void swap_column(const SwapLists& S, int nb, double2* __restrict__ col, bool inverse) {
  const int lane = threadIdx.x & 31;
  double2 v[16];
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int e = s * 32 + lane;
    if (e < 2 * nb && S.dst[e] >= 0) v[s] = col[inverse ? S.dst[e] : S.src[e]];
  }
  __syncwarp();
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int e = s * 32 + lane;
    if (e < 2 * nb && S.dst[e] >= 0) col[inverse ? S.src[e] : S.dst[e]] = v[s];
  }
}
