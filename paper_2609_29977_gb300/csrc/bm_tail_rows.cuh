// Register-resident variant of the tail tasks (Alg. 1, steps 1-3) for block
// sizes up to 32: a team of TS = next power of two >= NB lanes (at most one
// warp) handles one chain position, lane i holding row i of every block it
// works on in registers:
//   * the gathered Schur update D~_q -= X X^T streams the other rows of X
//     from shared memory (broadcast reads),
//   * the Cholesky of D~_q is right-looking with each column's entries
//     exchanged by warp shuffles (no shared memory, no barrier),
//   * the two coupling solves M L^{-T} reuse the shuffled columns of L,
//   * the fill -L_{b,q} L_{a,q}^T streams L_{a,q} from shared memory.
// D~ is kept with both triangles (each lane owns a full row), so the level
// workspace is read back row by row. Used for the FP32 tails of the mixed
// path, where the shared-memory variant is latency-bound.
#pragma once

#include "bm_team.cuh"

namespace bm {
namespace rows {

template <int NB>
struct Cfg {
  static constexpr int TS = NB <= 4 ? 4 : NB <= 8 ? 8 : NB <= 16 ? 16 : 32;
  // Blocks whose rows are groups of four floats move through shared memory
  // (factor_task_staged); the others (nb = 2, 3, 6) keep one staged block.
  static constexpr bool STAGED = NB % 4 == 0;
  // row stride of staged blocks without bank conflicts: an odd number of
  // 16-byte groups (rows read and written four floats at a time), or NB + 1
  static constexpr int LD = STAGED ? (NB / 4 % 2 ? NB : NB + 4) : NB + 1;
  static constexpr int BLK = NB * LD;               // one staged block
  static constexpr int SM = STAGED ? 4 * BLK : BLK; // per team
};

template <typename T>
__device__ __forceinline__ T shfl(unsigned mask, T v, int src, int width) {
  return __shfl_sync(mask, v, src, width);
}

// NB FP64 values addr(0), ..., addr(NB-1) rounded to FP32, every load of a
// chunk issued before its first conversion. The conversion is the hardware
// round-to-nearest (on this GPU's FP64 pipe, idle in these FP32 tasks; the
// same bits as the integer rounding d2f_rn, which a GPU test checks), so
// that no branch orders the loads: with the integer rounding's
// out-of-range branch after each value, each load waited for the data of
// the one before.
template <typename T, int NB, typename Addr>
__device__ __forceinline__ void load_to_t(T (&dst)[NB], Addr addr) {
  static_assert(sizeof(T) == sizeof(float), "FP32 tasks");
  constexpr int CH = NB <= 32 ? NB : 16;
#pragma unroll
  for (int j0 = 0; j0 < NB; j0 += CH) {
    double v[CH];
#pragma unroll
    for (int t = 0; t < CH; ++t)
      if (j0 + t < NB) v[t] = addr(j0 + t);
#pragma unroll
    for (int t = 0; t < CH; ++t)
      if (j0 + t < NB) dst[j0 + t] = __double2float_rn(v[t]);
  }
}

// Copy an NB x NB block (global, type T) into shared memory with the team
// (row stride Cfg<NB>::LD).
template <typename T, int NB, int TS>
__device__ __forceinline__ void stage(T *__restrict__ s, const T *__restrict__ g, int lane) {
#pragma unroll
  for (int e = lane; e < NB * NB; e += TS) {
    const int r = e / NB, c = e - r * NB;
    s[r * Cfg<NB>::LD + c] = g[e];
  }
}

// d[j] -= sum_k X[i][k] X[j][k] for all j, X staged in sX, row i = lane.
template <typename T, int NB>
__device__ __forceinline__ void syrk_row(T (&d)[NB], const T *__restrict__ sX, int ir) {
  constexpr int LD = Cfg<NB>::LD;
  T xi[NB];
#pragma unroll
  for (int k = 0; k < NB; ++k) xi[k] = sX[ir * LD + k];
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < NB; ++k) acc = fma_t<T>(xi[k], sX[j * LD + k], acc);
    d[j] -= acc;
  }
}

// Right-looking Cholesky on rows held by lanes (lane i has row i in d[]).
// On return d[j] (j <= i) is L_ij; rinv is 1/L_ii. Returns 1 + the first
// failing column (uniform over the team), 0 if all pivots are positive.
template <typename T, int NB, int TS>
__device__ __forceinline__ int chol_rows(T (&d)[NB], T &rinv, unsigned mask, int i) {
  int fail = 0;
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    T piv = shfl<T>(mask, d[j], j, TS);
    if (!pivot_ok(piv)) {
      if (!fail) fail = j + 1;
      piv = T(1);
    }
    const T r = rsqrt_t<T>(piv);
    if (i == j) {
      d[j] = piv * r;
      rinv = r;
    } else {
      d[j] *= r;
    }
#pragma unroll
    for (int k = j + 1; k < NB; ++k) {
      const T lkj = shfl<T>(mask, d[j], k, TS);
      d[k] = fma_t<T>(-d[j], lkj, d[k]);
    }
  }
  return fail;
}

// b := b L^{-T}, a := a L^{-T} for the rows held by this lane; L is
// distributed by rows over the team (lane k holds L_k* in lk[]).
template <typename T, int NB, int TS, bool TWO>
__device__ __forceinline__ void trsm_rows(T (&b)[NB], T (&a)[NB], const T (&lk)[NB], T rinv, unsigned mask) {
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    const T rj = shfl<T>(mask, rinv, j, TS);
    b[j] *= rj;
    if (TWO) a[j] *= rj;
#pragma unroll
    for (int k = j + 1; k < NB; ++k) {
      const T lkj = shfl<T>(mask, lk[j], k, TS);
      b[k] = fma_t<T>(-b[j], lkj, b[k]);
      if (TWO) a[k] = fma_t<T>(-a[j], lkj, a[k]);
    }
  }
}

// chol_rows and trsm_rows fused column by column: each entry L_kj that
// the Cholesky broadcasts also updates the coupling rows b (and a), which
// trsm_rows would broadcast a second time, and the inverse pivot 1/L_jj is
// the r every lane has just computed. The values and the order of the
// operations on d, b and a are those of chol_rows followed by trsm_rows.
template <typename T, int NB, int TS, bool TWO>
__device__ __forceinline__ int chol_trsm_rows(T (&d)[NB], T (&b)[NB], T (&a)[NB], T &rinv, unsigned mask, int i) {
  int fail = 0;
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    T piv = shfl<T>(mask, d[j], j, TS);
    if (!pivot_ok(piv)) {
      if (!fail) fail = j + 1;
      piv = T(1);
    }
    const T r = rsqrt_t<T>(piv);
    if (i == j) {
      d[j] = piv * r;
      rinv = r;
    } else {
      d[j] *= r;
    }
    b[j] *= r;
    if (TWO) a[j] *= r;
#pragma unroll
    for (int k = j + 1; k < NB; ++k) {
      const T lkj = shfl<T>(mask, d[j], k, TS);
      d[k] = fma_t<T>(-d[j], lkj, d[k]);
      b[k] = fma_t<T>(-b[j], lkj, b[k]);
      if (TWO) a[k] = fma_t<T>(-a[j], lkj, a[k]);
    }
  }
  return fail;
}

// 16-byte asynchronous copy, global to shared memory through L2.
__device__ __forceinline__ void cp_async16(void *s, const void *g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void *s, const void *g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all groups but the newest have arrived
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// An NB x NB float block, global (contiguous) <-> shared memory (row stride
// LD), 16 bytes per access and contiguous over the team.
template <int NB, int TS, int LD = Cfg<NB>::LD>
__device__ __forceinline__ void block_in(float *__restrict__ s, const float *__restrict__ g, int lane) {
#pragma unroll
  for (int e = lane; e < NB * NB / 4; e += TS) {
    const int r = 4 * e / NB, c = 4 * e - r * NB;
    cp_async16(s + r * LD + c, g + 4 * e);
  }
}
template <int NB, int TS, int LD = Cfg<NB>::LD>
__device__ __forceinline__ void block_out(float *__restrict__ g, const float *__restrict__ s, int lane) {
#pragma unroll
  for (int e = lane; e < NB * NB / 4; e += TS) {
    const int r = 4 * e / NB, c = 4 * e - r * NB;
    reinterpret_cast<float4 *>(g)[e] = *reinterpret_cast<const float4 *>(s + r * LD + c);
  }
}
// An FP64 input block, rounded to FP32, into shared memory: two doubles per
// load, contiguous over the team, all loads before the first conversion (the
// hardware rounding, see load_to_t). LOWER: only pairs that reach the lower triangle.
// Single loads where the caller's array is not 16-byte aligned (a batch takes
// pointers that the host does not see).
template <int NB, int TS, bool LOWER, int LD = Cfg<NB>::LD>
__device__ __forceinline__ void block_in_d(float *__restrict__ s, const double *__restrict__ g, int lane) {
  // 9 loads in flight per lane (all of a 24 x 24 block, half of a 48 x 48 one)
  constexpr int Q = NB * NB / 2, M = (Q + TS - 1) / TS, CH = M < 9 ? M : 9;
  if ((reinterpret_cast<unsigned long long>(g) & 15) != 0) {
#pragma unroll 1
    for (int e = lane; e < NB * NB; e += TS) {
      const int r = e / NB, c = e - r * NB;
      if (!LOWER || c <= r) s[r * LD + c] = __double2float_rn(g[e]);
    }
    return;
  }
#pragma unroll
  for (int t0 = 0; t0 < M; t0 += CH) {
    double2 v[CH];
#pragma unroll
    for (int t = 0; t < CH; ++t) {
      const int e = lane + (t0 + t) * TS, r = 2 * e / NB, c = 2 * e - r * NB;
      if (e < Q && (!LOWER || c <= r)) v[t] = reinterpret_cast<const double2 *>(g)[e];
    }
#pragma unroll
    for (int t = 0; t < CH; ++t) {
      const int e = lane + (t0 + t) * TS, r = 2 * e / NB, c = 2 * e - r * NB;
      if (e < Q && (!LOWER || c <= r))
        *reinterpret_cast<float2 *>(s + r * LD + c) =
            make_float2(__double2float_rn(v[t].x), __double2float_rn(v[t].y));
    }
  }
}
// A row of a staged block <-> registers.
template <int NB>
__device__ __forceinline__ void row_in(float (&d)[NB], const float *__restrict__ row) {
#pragma unroll
  for (int g = 0; g < NB / 4; ++g) {
    const float4 v = reinterpret_cast<const float4 *>(row)[g];
    d[4 * g] = v.x;
    d[4 * g + 1] = v.y;
    d[4 * g + 2] = v.z;
    d[4 * g + 3] = v.w;
  }
}
template <int NB>
__device__ __forceinline__ void row_out(float *__restrict__ row, const float (&d)[NB]) {
#pragma unroll
  for (int g = 0; g < NB / 4; ++g)
    reinterpret_cast<float4 *>(row)[g] = make_float4(d[4 * g], d[4 * g + 1], d[4 * g + 2], d[4 * g + 3]);
}
// sum_k a[k] row[k], k in increasing order (row staged, read by all lanes).
template <int NB>
__device__ __forceinline__ float row_dot(const float (&a)[NB], const float *__restrict__ row) {
  float acc = 0.0f;
#pragma unroll
  for (int g = 0; g < NB / 4; ++g) {
    const float4 v = reinterpret_cast<const float4 *>(row)[g];
    acc = fmaf(a[4 * g], v.x, acc);
    acc = fmaf(a[4 * g + 1], v.y, acc);
    acc = fmaf(a[4 * g + 2], v.z, acc);
    acc = fmaf(a[4 * g + 3], v.w, acc);
  }
  return acc;
}

// One task of level lvl with register-resident rows, every block moved
// between global and shared memory contiguously (16 bytes per lane) and
// between shared memory and the lanes' rows without bank conflicts. With a
// lane per row, rows loaded and stored straight from global memory put each
// lane of an access on a line of its own: for nb = 24 about 3500 L1 tag
// cycles per task of level 0, which took most of the level's time. The
// float blocks of a task (D~, both neighbours' couplings, the fill) are
// requested together, before anything waits for one of them.
// S = 512, N = 128, nb = 24: level 0 405 -> 252 us, level 1 321 -> 214,
// FP32+IR factor and solve 4304 -> 3919 us; S = N = 64, nb = 12: 288 -> 277.
// What bounds level 0 now is the conversion of
// the FP64 inputs (FP64 pipe 44%) and the columns' shuffle chains.
// The arithmetic and its order are those of factor_task_plain.
// FUSED: the Cholesky and the coupling solves in one column loop
// (chol_trsm_rows; the grid-wide level kernel) or one after the other (the
// per-tail top kernel and the batched form, whose register budget the
// fused loop would exceed). Both give the same bits.
// buf: Cfg<NB>::SM floats per team, 16-byte aligned.
template <int NB, bool FUSED>
__device__ __forceinline__ void factor_task_staged(const TailView<float> &v, float *buf, int lane, unsigned mask,
                                                   int s, int q, int lvl, bool elim) {
  constexpr int TS = Cfg<NB>::TS, NB2 = NB * NB, LD = Cfg<NB>::LD, BLK = Cfg<NB>::BLK;
  float *b0 = buf, *b1 = buf + BLK, *b2 = b1 + BLK, *b3 = b2 + BLK;
  const int N = v.N;
  const size_t sb = (size_t)s * N;
  const int i = lane;
  const bool act = i < NB;
  const int ir = act ? i : 0;
  int pl = 0, pr = 0;
  if (lvl >= 1) {
    const int h = 1 << (lvl - 1);
    if (q < N) {
      pl = q - h;
      if (q + h <= N - 1) pr = q + h;
    } else {
      const int m = ((N - 1) >> (lvl - 1)) << (lvl - 1);
      if (ctz32(m) == lvl - 1) pl = m;
    }
  }
  const int hh = 1 << lvl;
  const bool hasA = q > hh;
  const int a = q - hh;
  const bool inputB = lvl == 0 || q == N - 1;   // M_{b,q} is an input block (E^T)
  if (lvl >= 2) block_in<NB, TS>(b0, v.Dt + (sb + (N - q)) * NB2, lane);
  if (pl) block_in<NB, TS>(b1, v.Lr + (sb + (N - pl)) * NB2, lane);
  if (pr) block_in<NB, TS>(b2, v.Ll + (sb + (N - pr)) * NB2, lane);
  if (elim && !inputB) block_in<NB, TS>(b3, v.W + (sb + (N - q)) * NB2, lane);
  if (lvl <= 1) block_in_d<NB, TS, true>(b0, v.D + (sb + (N - q)) * NB2, lane);
  if (lvl == 0 && hasA) block_in_d<NB, TS, false>(b2, v.E + ((size_t)s * (N - 1) + (N - q)) * NB2, lane);
  cp_async_wait();
  __syncwarp(mask);
  float d[NB];
  if (lvl <= 1) {
#pragma unroll
    for (int j = 0; j < NB; ++j) d[j] = j <= ir ? b0[ir * LD + j] : b0[j * LD + ir];
  } else {
    row_in<NB>(d, b0 + ir * LD);
  }
  if (pl) {
    float x[NB];
    row_in<NB>(x, b1 + ir * LD);
#pragma unroll
    for (int j = 0; j < NB; ++j) d[j] -= row_dot<NB>(x, b1 + j * LD);
  }
  if (pr) {
    float x[NB];
    row_in<NB>(x, b2 + ir * LD);
#pragma unroll
    for (int j = 0; j < NB; ++j) d[j] -= row_dot<NB>(x, b2 + j * LD);
  }
  __syncwarp(mask);   // the staged inputs have been read
  if (!elim) {
    if (act) row_out<NB>(b0 + i * LD, d);
    __syncwarp(mask);
    block_out<NB, TS>(v.Dt + (sb + (N - q)) * NB2, b0, lane);
    __syncwarp(mask);
    return;
  }
  // couplings: rows i of M_{b,q} and M_{a,q}
  float b[NB], av[NB];
  if (inputB) {
    const double *Eb = v.E + ((size_t)s * (N - 1) + (N - q - 1)) * NB2;   // M_{b,q} = E^T: contiguous over the lanes
    load_to_t<float, NB>(b, [&](int k) { return Eb[k * NB + ir]; });
  } else {
    row_in<NB>(b, b3 + ir * LD);
  }
  if (hasA) {
    if (lvl == 0) {
      row_in<NB>(av, b2 + ir * LD);
    } else {
      const float *Wa = v.W + (sb + (N - a)) * NB2;   // M_{a,q} = W[a]^T: contiguous over the lanes
#pragma unroll
      for (int k = 0; k < NB; ++k) av[k] = Wa[k * NB + ir];
    }
  } else {
#pragma unroll
    for (int k = 0; k < NB; ++k) av[k] = 0.0f;
  }
  float rinv = 1.0f;
  int fail;
  if constexpr (FUSED) {
    // one instantiation for both cases: without a left neighbour av is zero
    // and stays +0 through the updates
    fail = chol_trsm_rows<float, NB, TS, true>(d, b, av, rinv, mask, i);
  } else {
    fail = chol_rows<float, NB, TS>(d, rinv, mask, i);
    if (hasA)
      trsm_rows<float, NB, TS, true>(b, av, d, rinv, mask);
    else
      trsm_rows<float, NB, TS, false>(b, av, d, rinv, mask);
  }
  if (i == 0 && fail) report_not_spd(v.status, s, N + 1 - q);
  if (act) {
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (j > i) d[j] = 0.0f;
    row_out<NB>(b0 + i * LD, d);
    row_out<NB>(b1 + i * LD, b);
    row_out<NB>(b2 + i * LD, av);
    v.invd[(sb + (N - q)) * NB + i] = rinv;
  }
  __syncwarp(mask);
  block_out<NB, TS>(v.Ld + (sb + (N - q)) * NB2, b0, lane);
  block_out<NB, TS>(v.Lr + (sb + (N - q)) * NB2, b1, lane);
  block_out<NB, TS>(v.Ll + (sb + (N - q)) * NB2, b2, lane);
  if (hasA) {
    // fill M_{b,a} = -L_{b,q} L_{a,q}^T (rows of L_{a,q} in b2)
    if (act) {
#pragma unroll
      for (int g = 0; g < NB / 4; ++g) {
        float w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = -row_dot<NB>(b, b2 + (4 * g + e) * LD);
        reinterpret_cast<float4 *>(b3 + i * LD)[g] = make_float4(w[0], w[1], w[2], w[3]);
      }
    }
    __syncwarp(mask);
    block_out<NB, TS>(v.W + (sb + (N - a)) * NB2, b3, lane);
  }
  __syncwarp(mask);
}

// One task of level lvl with register-resident rows loaded and stored
// straight from global memory (block sizes without groups of four).
template <typename T, int NB, bool FUSED = false>
__device__ __forceinline__ void factor_task_plain(const TailView<T> &v, T *sX, int lane, unsigned mask, int s, int q,
                                                 int lvl, bool elim) {
  constexpr int TS = Cfg<NB>::TS, NB2 = NB * NB;
  const int N = v.N;
  const size_t sb = (size_t)s * N;
  const int i = lane;
  const bool act = i < NB;
  const int ir = act ? i : 0;
  T d[NB];
  if (lvl <= 1) {
    const double *Dq = v.D + (sb + (N - q)) * NB2;
    load_to_t<T, NB>(d, [&](int j) { return j <= ir ? Dq[ir * NB + j] : Dq[j * NB + ir]; });
  } else {
    const T *Dq = v.Dt + (sb + (N - q)) * NB2 + ir * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) d[j] = Dq[j];
  }
  if (lvl >= 1) {
    const int h = 1 << (lvl - 1);
    int pl = 0, pr = 0;
    if (q < N) {
      pl = q - h;
      if (q + h <= N - 1) pr = q + h;
    } else {
      const int m = ((N - 1) >> (lvl - 1)) << (lvl - 1);
      if (ctz32(m) == lvl - 1) pl = m;
    }
    if (pl) {
      stage<T, NB, TS>(sX, v.Lr + (sb + (N - pl)) * NB2, lane);
      __syncwarp(mask);
      syrk_row<T, NB>(d, sX, ir);
      __syncwarp(mask);
    }
    if (pr) {
      stage<T, NB, TS>(sX, v.Ll + (sb + (N - pr)) * NB2, lane);
      __syncwarp(mask);
      syrk_row<T, NB>(d, sX, ir);
      __syncwarp(mask);
    }
  }
  if (!elim) {
    if (act) {
      T *o = v.Dt + (sb + (N - q)) * NB2 + i * NB;
#pragma unroll
      for (int j = 0; j < NB; ++j) o[j] = d[j];
    }
    return;
  }
  // couplings: rows i of M_{b,q} and M_{a,q}
  const int hh = 1 << lvl;
  const bool hasA = q > hh;
  const int a = q - hh;
  T b[NB], av[NB];
  if (lvl == 0 || q == N - 1) {
    const double *Eb = v.E + ((size_t)s * (N - 1) + (N - q - 1)) * NB2;   // M_{b,q} = E^T
    load_to_t<T, NB>(b, [&](int k) { return Eb[k * NB + ir]; });
  } else {
    const T *Wb = v.W + (sb + (N - q)) * NB2 + ir * NB;
#pragma unroll
    for (int k = 0; k < NB; ++k) b[k] = Wb[k];
  }
  if (hasA) {
    if (lvl == 0) {
      const double *Ea = v.E + ((size_t)s * (N - 1) + (N - q)) * NB2 + ir * NB;
      load_to_t<T, NB>(av, [&](int k) { return Ea[k]; });
    } else {
      const T *Wa = v.W + (sb + (N - a)) * NB2;   // M_{a,q} = W[a]^T
#pragma unroll
      for (int k = 0; k < NB; ++k) av[k] = Wa[k * NB + ir];
    }
  } else {
#pragma unroll
    for (int k = 0; k < NB; ++k) av[k] = T(0);
  }
  T rinv = T(1);
  int fail;
  if constexpr (FUSED) {
    // one instantiation for both cases: without a left neighbour av is zero
    // and stays +0 through the updates
    fail = chol_trsm_rows<T, NB, TS, true>(d, b, av, rinv, mask, i);
  } else {
    fail = chol_rows<T, NB, TS>(d, rinv, mask, i);
    if (hasA)
      trsm_rows<T, NB, TS, true>(b, av, d, rinv, mask);
    else
      trsm_rows<T, NB, TS, false>(b, av, d, rinv, mask);
  }
  if (i == 0 && fail) report_not_spd(v.status, s, N + 1 - q);
  if (act) {
    T *Ld = v.Ld + (sb + (N - q)) * NB2 + i * NB;
    T *Lb = v.Lr + (sb + (N - q)) * NB2 + i * NB;
    T *La = v.Ll + (sb + (N - q)) * NB2 + i * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      Ld[j] = j <= i ? d[j] : T(0);
      Lb[j] = b[j];
      La[j] = av[j];
    }
    v.invd[(sb + (N - q)) * NB + i] = rinv;
  }
  if (hasA) {
    // fill M_{b,a} = -L_{b,q} L_{a,q}^T: stage the rows of L_{a,q}
    constexpr int LD = Cfg<NB>::LD;
    if (act) {
#pragma unroll
      for (int k = 0; k < NB; ++k) sX[i * LD + k] = av[k];
    }
    __syncwarp(mask);
    if (act) {
      T *Wo = v.W + (sb + (N - a)) * NB2 + i * NB;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        T acc = T(0);
#pragma unroll
        for (int k = 0; k < NB; ++k) acc = fma_t<T>(b[k], sX[j * LD + k], acc);
        Wo[j] = -acc;
      }
    }
    __syncwarp(mask);
  }
}

template <typename T, int NB, bool FUSED = false>
__device__ __forceinline__ void factor_task_rows(const TailView<T> &v, T *sX, int lane, unsigned mask, int s, int q,
                                                 int lvl, bool elim) {
  if constexpr (Cfg<NB>::STAGED)
    factor_task_staged<NB, FUSED>(v, sX, lane, mask, s, q, lvl, elim);
  else
    factor_task_plain<T, NB, FUSED>(v, sX, lane, mask, s, q, lvl, elim);
}

// x_1 of tail s: last update and L_{i,1} with register rows, then F_{i,1} =
// C_{i,1} L_{i,1}^{-T} and U_i = F F^T in FP64. sbuf: nr*NB doubles followed
// by NB*NB + NB values of type T.
template <typename T, int NB>
__device__ __forceinline__ void x1_task_rows(const TailView<T> &v, void *sbuf, int lane, unsigned mask, int s) {
  constexpr int TS = Cfg<NB>::TS, NB2 = NB * NB;
  const int N = v.N, nr = v.nr, Lc = v.Lc;
  const size_t sb = (size_t)s * N;
  constexpr int LD = Cfg<NB>::LD;
  double *sC = (double *)sbuf;
  T *sL = (T *)(sC + nr * NB), *sInv = sL + NB * LD;
  const int i = lane;
  const bool act = i < NB;
  const int ir = act ? i : 0;
  T d[NB];
  if (Lc <= 1) {
    const double *Dq = v.D + sb * NB2;
    load_to_t<T, NB>(d, [&](int j) { return j <= ir ? Dq[ir * NB + j] : Dq[j * NB + ir]; });
  } else {
    const T *Dq = v.Dt + sb * NB2 + ir * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) d[j] = Dq[j];
  }
  if (Lc >= 1) {
    const int m = 1 << (Lc - 1);
    stage<T, NB, TS>(sL, v.Lr + (sb + (N - m)) * NB2, lane);
    __syncwarp(mask);
    syrk_row<T, NB>(d, sL, ir);
    __syncwarp(mask);
  }
  T rinv = T(1);
  const int fail = chol_rows<T, NB, TS>(d, rinv, mask, i);
  if (i == 0 && fail) report_not_spd(v.status, s, 1);
  if (act) {
    T *Ld = v.Ld + sb * NB2 + i * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      Ld[j] = j <= i ? d[j] : T(0);
      sL[i * LD + j] = j <= i ? d[j] : T(0);
      v.Lr[sb * NB2 + i * NB + j] = T(0);
      v.Ll[sb * NB2 + i * NB + j] = T(0);
    }
    v.invd[sb * NB + i] = rinv;
    sInv[i] = rinv;
  }
  for (int e = lane; e < nr * NB; e += TS) sC[e] = v.C[(size_t)s * nr * NB + e];
  __syncwarp(mask);
  // F = C L^{-T} in FP64, one row of C per lane (column sweep within the row)
  for (int c = lane; c < nr; c += TS) {
    double f[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) f[k] = sC[c * NB + k];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      f[j] *= to_d<T>(sInv[j]);
#pragma unroll
      for (int k = j + 1; k < NB; ++k) f[k] = fma(-f[j], to_d<T>(sL[k * LD + j]), f[k]);
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      sC[c * NB + k] = f[k];
      v.F[(size_t)s * nr * NB + c * NB + k] = f[k];
    }
  }
  __syncwarp(mask);
  double *Us = v.U + (size_t)s * nr * nr;
  for (int e = lane; e < nr * nr; e += TS) {
    const int a = e / nr, b = e - a * nr;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) acc = fma(sC[a * NB + k], sC[b * NB + k], acc);
    Us[e] = acc;
  }
}

template <typename T, int NB>
__host__ __device__ constexpr size_t x1_rows_bytes(int nr) {
  return (size_t)nr * NB * sizeof(double) + (NB * Cfg<NB>::LD + NB) * sizeof(T);
}

}  // namespace rows
}  // namespace bm

namespace bm {
namespace rows {

// Grid-wide level with register rows: tasks of all tails, eliminated
// positions first; TS lanes per task, 128 threads per CTA.
template <typename T, int NB>
__global__ void __launch_bounds__(128, 4) k_level_rows(TailView<T> v, int lvl) {
  constexpr int TS = Cfg<NB>::TS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int team = threadIdx.x / TS, lane = threadIdx.x % TS;
  const unsigned mask = TS == 32 ? 0xffffffffu : (((1u << TS) - 1u) << ((threadIdx.x & 31) / TS * TS));
  T *sX = (T *)smem_raw + team * Cfg<NB>::SM;
  const int N = v.N, S = v.S;
  const int E = level_elims(N, lvl);
  const int G = lvl == 0 ? 0 : ((N - 1) >> (lvl + 1)) + 1;
  const long g = (long)blockIdx.x * (blockDim.x / TS) + team;
  pdl_wait();
  if (g < (long)S * (E + G)) {
    int s, q;
    bool elim;
    if (g < (long)S * E) {
      s = (int)(g / E);
      q = (2 * (int)(g - (long)s * E) + 1) << lvl;
      elim = true;
    } else {
      const long g2 = g - (long)S * E;
      s = (int)(g2 / G);
      const int j = (int)(g2 - (long)s * G);
      q = j < G - 1 ? (j + 1) << (lvl + 1) : N;
      elim = false;
    }
    factor_task_rows<T, NB, true>(v, sX, lane, mask, s, q, lvl, elim);
  }
  pdl_trigger();
}

// Teams of the top kernel's CTA. Its levels have at most four positions each;
// with many tails the further teams idle in most of them and cost the
// registers and shared memory of other tails.
// nb = 24 and 32 take 255 registers (at 128, for four CTAs of four teams per
// SM, they spill 300 to 700 bytes, whatever S is). So that all tails stay on
// the SMs at once there are four teams up to two tails per SM (304), two up to
// four (608), one beyond. Factor, us, four teams at 128 registers -> this
// rule: nb = 24: S = 150, N = 6 109 -> 91; S = 304, N = 64 367 -> 352; S = 512, N = 6
// 144 -> 109, N = 128 882 -> 867; S = 609, N = 20 334 -> 252; nb = 32: S = 4, N = 8
// 171 -> 150; S = 304, N = 8 258 -> 212; S = 512, N = 6 397 -> 222; S = 1000, N = 12
// 710 -> 558. Slower between three tails per SM and more levels: nb = 32,
// S = 400, N = 20 412 -> 445, N = 64 848 -> 867 (four teams uncapped: S = 440,
// N = 20 434 -> 510). Two teams from S = 153 on: S = 153, N = 8 92 -> 101 (nb = 24).
template <int NB>
inline int top_teams(int S) {
  return NB <= 16 || S <= 2 * 152 ? 4 : S <= 4 * 152 ? 2 : 1;
}

// Top levels lvl0..Lc-1 and x_1 of one tail per CTA. Four CTAs per SM for the
// smaller blocks, which fit 128 registers: left to itself the compiler takes
// up to 254 (factor of S = 1000, N = 12, nb = 16: 136 us, uncapped 161).
template <typename T, int NB>
__global__ void __launch_bounds__(128, NB <= 16 ? 4 : 1) k_top_rows(TailView<T> v, int lvl0) {
  constexpr int TS = Cfg<NB>::TS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int team = threadIdx.x / TS, lane = threadIdx.x % TS, teams = blockDim.x / TS;
  const unsigned mask = TS == 32 ? 0xffffffffu : (((1u << TS) - 1u) << ((threadIdx.x & 31) / TS * TS));
  T *sX = (T *)smem_raw + team * Cfg<NB>::SM;
  const int N = v.N, s = blockIdx.x;
  pdl_wait();
  for (int lvl = lvl0; lvl < v.Lc; ++lvl) {
    const int E = level_elims(N, lvl);
    const int G = lvl == 0 ? 0 : ((N - 1) >> (lvl + 1)) + 1;
    for (int t = team; t < E + G; t += teams) {
      const bool elim = t < E;
      const int q = elim ? (2 * t + 1) << lvl : (t - E < G - 1 ? (t - E + 1) << (lvl + 1) : N);
      factor_task_rows<T, NB>(v, sX, lane, mask, s, q, lvl, elim);
    }
    __syncthreads();
  }
  if (team == 0) x1_task_rows<T, NB>(v, smem_raw, lane, mask, s);
  pdl_trigger();
}

template <typename T, int NB>
cudaError_t prepare_rows() {
  cudaError_t e = cudaFuncSetAttribute(k_level_rows<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_top_rows<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
}

template <typename T, int NB>
void launch_tail_rows(const TailView<T> &v, cudaStream_t st) {
  constexpr int TS = Cfg<NB>::TS;
  const int Tl = top_level(v.N);
  const int tpc = 128 / TS;
  for (int l = 0; l < Tl; ++l) {
    const int E = level_elims(v.N, l);
    const int G = l == 0 ? 0 : ((v.N - 1) >> (l + 1)) + 1;
    const long tasks = (long)v.S * (E + G);
    const long blocks = (tasks + tpc - 1) / tpc;
    launch_pdl(k_level_rows<T, NB>, (unsigned)blocks, 128, (size_t)tpc * Cfg<NB>::SM * sizeof(T), st, v, l);
  }
  const int teams = top_teams<NB>(v.S);
  size_t smem = (size_t)teams * Cfg<NB>::SM * sizeof(T);
  const size_t x1b = x1_rows_bytes<T, NB>(v.nr);
  if (x1b > smem) smem = x1b;
  launch_pdl(k_top_rows<T, NB>, (unsigned)v.S, teams * TS, smem, st, v, Tl);
}

}  // namespace rows
}  // namespace bm
