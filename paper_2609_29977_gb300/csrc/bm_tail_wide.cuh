// FP32 tail tasks (Alg. 1, steps 1-3) for block sizes above 32 (nb = 48): a
// team of three warps per chain position, the blocks in shared memory, and
// loops of a few hundred instructions:
//   * Schur updates and fill: a 4 x 6 tile of the 48 x 48 product per lane
//     (10 shared loads of 16 bytes per 96 FMAs; of a symmetric update only
//     the tile entries that reach the lower triangle),
//   * Cholesky in panels of four columns, left-looking, a row per lane, the
//     4 x 4 pivot block factored by every lane (two barriers per panel),
//   * both coupling solves at once, a row of M_b or M_a per lane, eight
//     columns at a time, no barrier.
// Every element's operations and their order are those of the right-looking
// register-row tasks (bm_tail_rows.cuh): d_ik and x_k lose their products in
// increasing column order, each by one FMA, and are then scaled; dot
// products of updates start from zero.
//
// A lane per row with rows in registers needs fully unrolled code (about
// 12000 FMAs for nb = 48): the level kernel then waited on instruction fetch
// (3.5 of 8 stall cycles per issue) at 6 tasks per SM. Here it is 80 registers
// and seven tasks per SM. S = 512, N = 256, nb = 48: FP32+IR factor and solve
// 26.6 -> 19.0 ms; level 0 of it 3661 us before, S = 128, N = 128 (an eighth of
// its tasks) 249 us now; a batch of 16 systems 8.8 -> 6.6 ms. The level kernel
// issues in half of the cycles (FMA pipe 35%, barriers and shared-memory
// latency behind it).
#pragma once

#include "bm_tail_rows.cuh"

namespace bm {
namespace rows {

template <int NB>
struct WCfg {
  static_assert(NB == 48, "4 x 6 tiles on a 12 x 8 grid of lanes");
  static constexpr int TS = 96;
  // row stride: an odd number of 16-byte groups (no bank conflicts)
  static constexpr int LD = NB + 4;
  static constexpr int SM = NB * LD;
  // per team (floats): M_b / L_b, M_a / L_a, D~ / L, inverse pivots, two 4 x 4 pivot blocks
  static constexpr int ELEMS = 3 * SM + NB + 32;
};

__device__ __forceinline__ void team_bar(int id) { asm volatile("bar.sync %0, 96;" ::"r"(id) : "memory"); }

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// acc - x . l over four columns in order.
__device__ __forceinline__ float sub_dot4(float acc, const float4 &x, const float4 &l) {
  acc = fmaf(-x.x, l.x, acc);
  acc = fmaf(-x.y, l.y, acc);
  acc = fmaf(-x.z, l.z, acc);
  return fmaf(-x.w, l.w, acc);
}

// Cholesky of the block in sL (lower triangle read): on return L below and
// zeros above the diagonal within each row's panels up to its own, and the
// inverse pivots in sInv. The return value (1 + the first failed column, 0 if
// none) is that of lane NB - 1.
template <int NB>
__device__ __forceinline__ int chol_w(float *sL, float *sInv, float *sP, int lane, int bar) {
  constexpr int LD = WCfg<NB>::LD;
  float *mine = sL + (lane < NB ? lane : 0) * LD;
  int fail = 0;
#pragma unroll 1
  for (int p = 0; p < NB / 4; ++p) {
    const int c0 = 4 * p, own = lane - c0;   // own: column of this row's pivot within the panel
    const bool on = lane < NB && own >= 0;
    float *pb = sP + (p & 1) * 16;
    float acc[4];
    if (on) {
      const float4 v = lds4(mine + c0);
      acc[0] = v.x;
      acc[1] = v.y;
      acc[2] = v.z;
      acc[3] = v.w;
#pragma unroll 2
      for (int j = 0; j < c0; j += 4) {
        const float4 x = lds4(mine + j);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e] = sub_dot4(acc[e], x, lds4(sL + (c0 + e) * LD + j));
      }
      if (own < 4) *reinterpret_cast<float4 *>(pb + 4 * own) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    }
    team_bar(bar);
    if (on) {
      float P[4][4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float4 v = lds4(pb + 4 * m);
        P[m][0] = v.x;
        P[m][1] = v.y;
        P[m][2] = v.z;
        P[m][3] = v.w;
      }
      float rinv = 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float piv = P[j][j];
        if (!pivot_ok(piv)) {
          if (!fail) fail = c0 + j + 1;
          piv = 1.0f;
        }
        const float r = rsqrt_t<float>(piv);
#pragma unroll
        for (int m = j + 1; m < 4; ++m) P[m][j] *= r;
#pragma unroll
        for (int m = j + 1; m < 4; ++m)
#pragma unroll
          for (int k = j + 1; k <= m; ++k) P[m][k] = fmaf(-P[m][j], P[k][j], P[m][k]);
        if (own == j) {
          acc[j] = piv * r;
          rinv = r;
        } else {
          acc[j] *= r;
        }
#pragma unroll
        for (int k = j + 1; k < 4; ++k) acc[k] = fmaf(-acc[j], P[k][j], acc[k]);
      }
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (k > own) acc[k] = 0.0f;
      *reinterpret_cast<float4 *>(mine + c0) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      if (own < 4) sInv[lane] = rinv;
    }
    team_bar(bar);
  }
  return fail;
}

// row := row L^{-T} for one row in shared memory (L row-major in sL).
template <int NB>
__device__ __forceinline__ void trsm_w(float *row, const float *sL, const float *sInv) {
  constexpr int LD = WCfg<NB>::LD;
#pragma unroll 1
  for (int k0 = 0; k0 < NB; k0 += 8) {
    float x[8];
    const float4 u = lds4(row + k0), w = lds4(row + k0 + 4);
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
    x[4] = w.x; x[5] = w.y; x[6] = w.z; x[7] = w.w;
#pragma unroll 2
    for (int j = 0; j < k0; j += 4) {
      const float4 v = lds4(row + j);
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = sub_dot4(x[e], v, lds4(sL + (k0 + e) * LD + j));
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      x[j] *= sInv[k0 + j];
#pragma unroll
      for (int k = j + 1; k < 8; ++k) x[k] = fmaf(-x[j], sL[(k0 + k) * LD + k0 + j], x[k]);
    }
    *reinterpret_cast<float4 *>(row + k0) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4 *>(row + k0 + 4) = make_float4(x[4], x[5], x[6], x[7]);
  }
}

// Products with rows of A and B: out(i, j, sum_k A_ik B_jk) for this lane's
// tile (rows r + 12 e, columns c + 8 f). LOWER: entries j <= i only.
template <int NB, bool LOWER, typename Out>
__device__ __forceinline__ void tile_product(const float *A, const float *B, int lane, Out out) {
  constexpr int LD = WCfg<NB>::LD;
  const int r = lane >> 3, c = lane & 7;
  float acc[4][6];
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int f = 0; f < 6; ++f) acc[e][f] = 0.0f;
#pragma unroll 1
  for (int k = 0; k < NB; k += 4) {
    float4 a[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) a[e] = lds4(A + (r + 12 * e) * LD + k);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const float4 b = lds4(B + (c + 8 * f) * LD + k);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (!LOWER || 8 * f <= 12 * e + 11) {
          acc[e][f] = fmaf(a[e].x, b.x, acc[e][f]);
          acc[e][f] = fmaf(a[e].y, b.y, acc[e][f]);
          acc[e][f] = fmaf(a[e].z, b.z, acc[e][f]);
          acc[e][f] = fmaf(a[e].w, b.w, acc[e][f]);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int f = 0; f < 6; ++f)
      if (!LOWER || (8 * f <= 12 * e + 11 && c + 8 * f <= r + 12 * e)) out(r + 12 * e, c + 8 * f, acc[e][f]);
}

// The transpose of an NB x NB block into shared memory: columns are loaded
// contiguously over the lanes and written four entries of a row at a time.
template <int NB, typename S>
__device__ __forceinline__ void block_in_t(float *__restrict__ s, const S *__restrict__ g, int lane) {
  constexpr int LD = WCfg<NB>::LD;
  const int i = lane % NB, half = lane / NB;
#pragma unroll
  for (int t = 0; t < NB / 4; t += 6) {
    S v[3][4];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int e = 0; e < 4; ++e) v[u][e] = g[(4 * (t + 2 * u + half) + e) * NB + i];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      float4 w;
      if constexpr (sizeof(S) == 8)
        w = make_float4(__double2float_rn(v[u][0]), __double2float_rn(v[u][1]), __double2float_rn(v[u][2]),
                        __double2float_rn(v[u][3]));
      else
        w = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
      *reinterpret_cast<float4 *>(s + i * LD + 4 * (t + 2 * u + half)) = w;
    }
  }
}

// The lower triangle of a staged block to global memory, zeros above it.
template <int NB>
__device__ __forceinline__ void block_out_lower(float *__restrict__ g, const float *__restrict__ s, int lane) {
  constexpr int LD = WCfg<NB>::LD;
#pragma unroll
  for (int e = lane; e < NB * NB / 4; e += WCfg<NB>::TS) {
    const int r = 4 * e / NB, c = 4 * e - r * NB;
    float4 v = lds4(s + r * LD + c);
    if (c > r) v.x = 0.0f;
    if (c + 1 > r) v.y = 0.0f;
    if (c + 2 > r) v.z = 0.0f;
    if (c + 3 > r) v.w = 0.0f;
    reinterpret_cast<float4 *>(g)[e] = v;
  }
}
template <int NB>
__device__ __forceinline__ void block_zero(float *__restrict__ g, int lane) {
#pragma unroll
  for (int e = lane; e < NB * NB / 4; e += WCfg<NB>::TS)
    reinterpret_cast<float4 *>(g)[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// One task of level lvl (sbuf: WCfg<NB>::ELEMS floats, 16-byte aligned).
template <int NB>
__device__ __forceinline__ void factor_task_w(const TailView<float> &v, float *sbuf, int lane, int bar, int s, int q,
                                              int lvl, bool elim) {
  constexpr int NB2 = NB * NB, LD = WCfg<NB>::LD, SM = WCfg<NB>::SM, TS = WCfg<NB>::TS;
  float *sB = sbuf, *sA = sB + SM, *sL = sA + SM, *sInv = sL + SM, *sP = sInv + NB;
  const int N = v.N;
  const size_t sb = (size_t)s * N;
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
  if (lvl >= 2) block_in<NB, TS, LD>(sL, v.Dt + (sb + (N - q)) * NB2, lane);
  if (pl) block_in<NB, TS, LD>(sB, v.Lr + (sb + (N - pl)) * NB2, lane);
  if (pr) block_in<NB, TS, LD>(sA, v.Ll + (sb + (N - pr)) * NB2, lane);
  if (lvl <= 1) block_in_d<NB, TS, true, LD>(sL, v.D + (sb + (N - q)) * NB2, lane);
  const double *Eb = v.E + ((size_t)s * (N - 1) + (N - q - 1)) * NB2;
  if (lvl == 0) {
    if (hasA) block_in_d<NB, TS, false, LD>(sA, v.E + ((size_t)s * (N - 1) + (N - q)) * NB2, lane);
    block_in_t<NB>(sB, Eb, lane);
  }
  cp_async_wait();
  team_bar(bar);
  if (pl) tile_product<NB, true>(sB, sB, lane, [&](int i, int j, float x) { sL[i * LD + j] -= x; });
  if (pr) tile_product<NB, true>(sA, sA, lane, [&](int i, int j, float x) { sL[i * LD + j] -= x; });
  if (lvl >= 1) team_bar(bar);   // the update is complete and its operands have been read
  if (!elim) {
    // the next level reads the lower triangle only
    block_out<NB, TS, LD>(v.Dt + (sb + (N - q)) * NB2, sL, lane);
    team_bar(bar);
    return;
  }
  if (lvl >= 1) {
    if (inputB)
      block_in_t<NB>(sB, Eb, lane);
    else
      block_in<NB, TS, LD>(sB, v.W + (sb + (N - q)) * NB2, lane);
    if (hasA) block_in_t<NB>(sA, v.W + (sb + (N - a)) * NB2, lane);   // M_{a,q} = W[a]^T
  }
  const int fail = chol_w<NB>(sL, sInv, sP, lane, bar);
  if (lane == NB - 1 && fail) report_not_spd(v.status, s, N + 1 - q);
  cp_async_wait();
  team_bar(bar);
  block_out_lower<NB>(v.Ld + (sb + (N - q)) * NB2, sL, lane);
  if (lane < NB) v.invd[(sb + (N - q)) * NB + lane] = sInv[lane];
  if (lane < NB)
    trsm_w<NB>(sB + lane * LD, sL, sInv);
  else if (hasA)
    trsm_w<NB>(sA + (lane - NB) * LD, sL, sInv);
  team_bar(bar);
  block_out<NB, TS, LD>(v.Lr + (sb + (N - q)) * NB2, sB, lane);
  if (hasA) {
    block_out<NB, TS, LD>(v.Ll + (sb + (N - q)) * NB2, sA, lane);
    // fill M_{b,a} = -L_{b,q} L_{a,q}^T, staged over L_qq
    tile_product<NB, false>(sB, sA, lane, [&](int i, int j, float x) { sL[i * LD + j] = -x; });
    team_bar(bar);
    block_out<NB, TS, LD>(v.W + (sb + (N - a)) * NB2, sL, lane);
  } else {
    block_zero<NB>(v.Ll + (sb + (N - q)) * NB2, lane);
  }
  team_bar(bar);
}

// x_1 of tail s: last update and L_{i,1}, then F_{i,1} = C_{i,1} L_{i,1}^{-T}
// and U_i = F F^T in FP64. sbuf: x1_w_bytes bytes.
template <int NB>
__host__ __device__ constexpr size_t x1_w_bytes(int nr) {
  return (size_t)nr * NB * sizeof(double) + (size_t)WCfg<NB>::ELEMS * sizeof(float);
}

template <int NB>
__device__ __forceinline__ void x1_task_w(const TailView<float> &v, void *sbuf, int lane, int bar, int s) {
  constexpr int NB2 = NB * NB, LD = WCfg<NB>::LD, SM = WCfg<NB>::SM, TS = WCfg<NB>::TS;
  const int N = v.N, nr = v.nr, Lc = v.Lc;
  const size_t sb = (size_t)s * N;
  double *sC = (double *)sbuf;
  float *sX = (float *)(sC + nr * NB), *sL = sX + 2 * SM, *sInv = sL + SM, *sP = sInv + NB;
  if (Lc > 1) block_in<NB, TS, LD>(sL, v.Dt + sb * NB2, lane);
  if (Lc >= 1) block_in<NB, TS, LD>(sX, v.Lr + (sb + (N - (1 << (Lc - 1)))) * NB2, lane);
  if (Lc <= 1) block_in_d<NB, TS, true, LD>(sL, v.D + sb * NB2, lane);
  for (int e = lane; e < nr * NB; e += TS) sC[e] = v.C[(size_t)s * nr * NB + e];
  cp_async_wait();
  team_bar(bar);
  if (Lc >= 1) {
    tile_product<NB, true>(sX, sX, lane, [&](int i, int j, float x) { sL[i * LD + j] -= x; });
    team_bar(bar);
  }
  const int fail = chol_w<NB>(sL, sInv, sP, lane, bar);
  if (lane == NB - 1 && fail) report_not_spd(v.status, s, 1);
  block_out_lower<NB>(v.Ld + sb * NB2, sL, lane);
  block_zero<NB>(v.Lr + sb * NB2, lane);
  block_zero<NB>(v.Ll + sb * NB2, lane);
  if (lane < NB) v.invd[sb * NB + lane] = sInv[lane];
  // F = C L^{-T}: eight columns at a time, one entry (c, k) per lane. The
  // eight lanes of a row stay the same for every group of columns, so the
  // row's earlier entries need a warp's synchronization only. A row per
  // lane, as before, ran 1128 dependent FP64 instructions on half a warp
  // (64 cycles each).
  const int rounds = (nr * 8 + TS - 1) / TS;
#pragma unroll 1
  for (int k0 = 0; k0 < NB; k0 += 8) {
    for (int t = 0; t < rounds; ++t) {
      const int p = lane + t * TS, kk = p & 7, c = p >> 3;
      const bool on = c < nr;
      double *row = sC + (on ? c : 0) * NB;
      const float *Lk = sL + (k0 + kk) * LD;
      double f = row[k0 + kk];
#pragma unroll 4
      for (int j = 0; j < k0; ++j) f = fma(-row[j], f2d_exact(Lk[j]), f);
      const double inv = f2d_exact(sInv[k0 + kk]);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (kk == j) f *= inv;
        const double fj = __shfl_sync(0xffffffffu, f, (threadIdx.x & 24) + j);
        if (kk > j) f = fma(-fj, f2d_exact(Lk[k0 + j]), f);
      }
      __syncwarp();
      if (on) row[k0 + kk] = f;
      __syncwarp();
    }
  }
  team_bar(bar);
  for (int e = lane; e < nr * NB; e += TS) v.F[(size_t)s * nr * NB + e] = sC[e];
  double *Us = v.U + (size_t)s * nr * nr;
  for (int e = lane; e < nr * nr; e += TS) {
    const int i = e / nr, j = e - i * nr;
    double acc = 0.0;
#pragma unroll 8
    for (int k = 0; k < NB; ++k) acc = fma(sC[i * NB + k], sC[j * NB + k], acc);
    Us[e] = acc;
  }
}

// Grid-wide level: one team per CTA (seven CTAs per SM).
template <int NB>
__global__ void __launch_bounds__(96, 7) k_level_rows_w(TailView<float> v, int lvl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = v.N, S = v.S, lane = threadIdx.x;
  const int E = level_elims(N, lvl);
  const int G = lvl == 0 ? 0 : ((N - 1) >> (lvl + 1)) + 1;
  const long g = blockIdx.x;
  int s, q;
  const bool elim = g < (long)S * E;
  if (elim) {
    s = (int)(g / E);
    q = (2 * (int)(g - (long)s * E) + 1) << lvl;
  } else {
    const long g2 = g - (long)S * E;
    s = (int)(g2 / G);
    const int j = (int)(g2 - (long)s * G);
    q = j < G - 1 ? (j + 1) << (lvl + 1) : N;
  }
  pdl_wait();
  factor_task_w<NB>(v, (float *)smem_raw, lane, 1, s, q, lvl, elim);
  pdl_trigger();
}

// Top levels lvl0..Lc-1 and x_1 of one tail per CTA.
template <int NB>
__global__ void __launch_bounds__(4 * 96) k_top_rows_w(TailView<float> v, int lvl0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TS = WCfg<NB>::TS;
  const int team = threadIdx.x / TS, lane = threadIdx.x - team * TS, teams = blockDim.x / TS;
  float *sb = (float *)smem_raw + team * WCfg<NB>::ELEMS;
  const int N = v.N, s = blockIdx.x;
  pdl_wait();
  for (int lvl = lvl0; lvl < v.Lc; ++lvl) {
    const int E = level_elims(N, lvl);
    const int G = lvl == 0 ? 0 : ((N - 1) >> (lvl + 1)) + 1;
    for (int t = team; t < E + G; t += teams) {
      const bool elim = t < E;
      const int q = elim ? (2 * t + 1) << lvl : (t - E < G - 1 ? (t - E + 1) << (lvl + 1) : N);
      factor_task_w<NB>(v, sb, lane, 1 + team, s, q, lvl, elim);
    }
    __syncthreads();
  }
  if (team == 0) x1_task_w<NB>(v, smem_raw, lane, 1, s);
  pdl_trigger();
}

template <int NB>
cudaError_t prepare_w() {
  cudaError_t e = cudaFuncSetAttribute(k_level_rows_w<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_top_rows_w<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

template <int NB>
void launch_tail_w(const TailView<float> &v, cudaStream_t st) {
  const int Tl = top_level(v.N);
  const size_t per = (size_t)WCfg<NB>::ELEMS * sizeof(float);
  for (int l = 0; l < Tl; ++l) {
    const int E = level_elims(v.N, l);
    const int G = l == 0 ? 0 : ((v.N - 1) >> (l + 1)) + 1;
    launch_pdl(k_level_rows_w<NB>, (unsigned)((long)v.S * (E + G)), 96, per, st, v, l);
  }
  // four teams per tail while every SM has a tail to itself, fewer with more
  // tails than that: the shared memory then holds more tails, and one
  // task's latency is what a level costs
  const int teams = v.S <= 152 ? 4 : v.S <= 304 ? 2 : 1;
  size_t smem = teams * per;
  const size_t x1b = x1_w_bytes<NB>(v.nr);
  if (x1b > smem) smem = x1b;
  launch_pdl(k_top_rows_w<NB>, (unsigned)v.S, teams * 96, smem, st, v, Tl);
}

}  // namespace rows
}  // namespace bm
