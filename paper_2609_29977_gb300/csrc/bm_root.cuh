// The root step of the factor (Alg. 1 steps 4-5) as device routines shared
// by the FP64 root kernel and the per-tail top kernel that can finish it:
// R~ = R - sum_i U_i entry by entry (one warp per entry, the library's
// fixed summation order root_sum_warp) and L_R = chol(R~) by one CTA.
#pragma once

#include <math.h>

#include "bm_internal.cuh"

namespace bm {

// global (n x n) := lower triangle of s, zeros above
__device__ __forceinline__ void cta_store_lower(double *__restrict__ g, const double *__restrict__ s, int n) {
  const int n2 = n * n;
  for (int e = threadIdx.x; e < n2; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    g[e] = (j <= i) ? s[e] : 0.0;
  }
}

// Lower-triangle element e -> (i, j) with j <= i.
__device__ __forceinline__ void tri_ij(int e, int &i, int &j) {
  int t = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((t + 1) * (t + 2) / 2 <= e) ++t;
  while (t * (t + 1) / 2 > e) --t;
  i = t;
  j = e - t * (t + 1) / 2;
}

// In-place lower Cholesky of the n x n block sA (lower triangle read);
// sInv[j] = 1 / L_jj. A pivot that is not positive and finite is replaced by
// 1 (so the launch finishes without NaNs) and the first such column + 1 is
// returned; 0 on success.
__device__ inline int cta_chol(double *sA, double *sInv, int n, int *sflag) {
  if (threadIdx.x == 0) *sflag = 0;
  for (int j = 0; j < n; ++j) {
    if (threadIdx.x == 0) {
      double d = sA[j * n + j];
      if (!(d > 0.0) || !(d < INFINITY)) {
        if (*sflag == 0) *sflag = j + 1;
        d = 1.0;
      }
      const double r = rsqrt(d);
      sA[j * n + j] = d * r;
      sInv[j] = r;
    }
    __syncthreads();
    const double r = sInv[j];
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) sA[i * n + j] *= r;
    __syncthreads();
    const int m = n - j - 1, ne = m * (m + 1) / 2;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      int a, b;
      tri_ij(e, a, b);
      const int i = j + 1 + a, k = j + 1 + b;
      sA[i * n + k] = fma(-sA[i * n + j], sA[k * n + j], sA[i * n + k]);
    }
    __syncthreads();
  }
  return *sflag;
}

// Entry e of the lower triangle of R~ = R - sum_i U_i, by one warp (all 32
// lanes), into Rt (both triangles).
__device__ __forceinline__ void root_entry(const double *U, const double *R, int S, int nr, int e, double *Rt) {
  int i, j;
  tri_ij(e, i, j);
  const double val = R[i * nr + j] - root_sum_warp(U, S, nr, i, j);
  if ((threadIdx.x & 31) == 0) {
    Rt[i * nr + j] = val;
    Rt[j * nr + i] = val;
  }
}

// L_R = chol(sR) (nr x nr in shared memory, followed by nr doubles of
// scratch) stored lower into LR. A failed pivot is reported at the root
// unless *engage (the mixed path's probe) takes over: then *on = engage
// and no failure is reported. Call with every thread of the CTA.
__device__ __forceinline__ void root_chol_store(double *sR, int nr, double *LR, Status *status, bool *engage,
                                                int *on) {
  __shared__ int sflag;
  const int fail = cta_chol(sR, sR + nr * nr, nr, &sflag);
  bool eng = false;
  if (engage) eng = *engage || fail;
  if (threadIdx.x == 0) {
    if (engage) *on = eng ? 1 : 0;
    if (fail && !eng) report_not_spd(status, -1, 0);
  }
  cta_store_lower(LR, sR, nr);
}

// Whether root_reduce_chol takes 32 entries at a time (nr >= 6), and the
// doubles of shared memory that it needs.
__host__ __device__ constexpr bool root_by_columns(int nr) { return nr * (nr + 1) / 2 > 16; }
__host__ __device__ constexpr int root_reduce_doubles(int nr) {
  return root_by_columns(nr) && nr * nr + nr < 32 * 33 ? 32 * 33 : nr * nr + nr;
}

// The whole root step by one CTA (a multiple of four, at most eight warps):
// every entry, then the Cholesky. Few entries: a warp per entry. More: one SM
// reads all of U here, so the lanes of a warp read neighbouring entries: warp w adds up the partial sums p_l of
// l = 4 w..4 w + 3 (and every 4 nw further on) for 32 entries at a time, sixteen loads in
// flight, and the 32 partial sums of an entry are then combined by a warp, all in
// the order of root_sum_warp. (With a warp per entry each load fetches 32
// sectors for 8 bytes of each: factor of S = 512, N = 6, nb = 24, nr = 24 521 us,
// 407 this way; nb = 16, nr = 6 113 and 105; nb = 4, nr = 4 31 and 35.)
// sm: root_reduce_doubles(nr).
__device__ __forceinline__ void root_reduce_chol(const double *U, const double *R, int S, int nr, double *Rt,
                                                 double *LR, Status *status, double *sm) {
  const int ne = nr * (nr + 1) / 2, nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t stride = (size_t)nr * nr;
  if (!root_by_columns(nr))
    for (int e = w; e < ne; e += nw) root_entry(U, R, S, nr, e, Rt);
  for (int e0 = 0; root_by_columns(nr) && e0 < ne; e0 += 32) {
    int i, j;
    tri_ij(e0 + lane < ne ? e0 + lane : ne - 1, i, j);
    const double *Ue = U + i * nr + j;
    for (int g = 4 * w; g < 32; g += 4 * nw) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      int s = g;
      for (; s + 99 < S; s += 128) {
        double v[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int u = 0; u < 4; ++u) v[k][u] = __ldcg(Ue + (size_t)(s + 32 * k + u) * stride);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[u] += v[k][u];
      }
      for (; s < S; s += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (s + u < S) acc[u] += __ldcg(Ue + (size_t)(s + u) * stride);
#pragma unroll
      for (int u = 0; u < 4; ++u) sm[(g + u) * 33 + lane] = acc[u];
    }
    __syncthreads();
    for (int q = w; q < 32 && e0 + q < ne; q += nw) {
      double acc = sm[lane * 33 + q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) {
        tri_ij(e0 + q, i, j);
        const double val = R[i * nr + j] - acc;
        Rt[i * nr + j] = val;
        Rt[j * nr + i] = val;
      }
    }
    __syncthreads();
  }
  __threadfence_block();
  __syncthreads();
  for (int k = threadIdx.x; k < nr * nr; k += blockDim.x) sm[k] = Rt[k];
  __syncthreads();
  root_chol_store(sm, nr, LR, status, nullptr, nullptr);
}

}  // namespace bm
