// FP32 tail substitutions of the mixed path for few tails: one CTA per tail,
// its vectors in shared memory, the factor's rows one position ahead in
// registers.
//
// With few tails the levels of a tail are a chain of latencies. In fwd_tail
// and bwd_tail a level pays a trip to L2 for the neighbours' vectors, one to
// memory for the factor's rows and, when a cluster shares the tail, a
// cluster barrier with its flush: 4 to 5 us for about 600 cycles of
// arithmetic. Here the vectors never leave the SM between levels, and the
// rows of a team's next position, which do not depend on the substitution,
// are requested as soon as the registers of the present one are free, across
// the barrier between levels.
// S = N = 64, nb = 12: factor and solve 284 -> 232 us; more shapes at
// chain_applies.
// The arithmetic of every row and its order are those of fwd_tail and
// bwd_tail (bm_mixed.cuh).
#pragma once

#include "bm_mixed.cuh"

namespace bm {
namespace mx {

template <int NB>
struct ChainCfg {
  static constexpr int TS = MCfg<NB>::TS, TEAMS = MCfg<NB>::TEAMS;
  // CTAs per SM that the registers allow (three rows of the factor per lane)
  static constexpr int CTAS = NB <= 32 ? 2 : 1;
  // for nb = 32 only with spilling (128 registers of 155 and 201): up to 152
  // tails get one CTA per SM instead. Solve, us: S = 4, N = 8 138 -> 130;
  // S = 64, N = 12 155 -> 146; S = 150, N = 64 410 -> 380
  static constexpr int FEW = NB == 32 ? 1 : CTAS;
  static constexpr size_t MAX_VEC = 96 * 1024;   // bytes of one tail's vectors
};

// Positions that a team walks one after another over all levels.
template <int NB>
inline int chain_rounds(int N) {
  const int Lc = chain_levels(N), T = ChainCfg<NB>::TEAMS;
  int r = 1;
  for (int l = 0; l < Lc; ++l) r += ((l == 0 ? N / 2 : ((N - 1) >> l) + 1) + T - 1) / T;
  return r;
}

// Whether a system's substitutions take this form: its tails fill the
// registers' CTAs at most once, and either the other form would have one CTA
// per tail as well (cluster size 1), or a team has few positions to walk, so
// that a cluster's further teams save less than its barriers cost. Solve with
// one or two corrections, clusters -> this form, us (rounds, cluster size):
//   S=64 N=64 nb=12 (9, 2) 143 -> 114      S=4 N=30 nb=16 (6, 8) 126 -> 98
//   S=100 N=160 nb=16 (20, 1) 346 -> 272   S=150 N=128 nb=24 (26, 1) 498 -> 381
//   S=140 N=100 nb=48 (42, 1) 1123 -> 913  S=280 N=100 nb=12 (18, 1) 379 -> 302
//   S=8 N=64 nb=24 (15, 8) 156 -> 160      S=20 N=200 nb=12 (24, 4) 168 -> 165
//   S=10 N=128 nb=24 (26, 8) 171 -> 225    S=40 N=60 nb=48 (25, 2) 411 -> 465
//   S=30 N=250 nb=32 (49, 4) 648 -> 1027   S=4 N=30 nb=32 (8, 8) 177 -> 166
//   S=4 N=40 nb=32 (12, 8) 189 -> 193
template <int NB>
inline bool chain_applies(int S, int N, int cluster) {
  return S <= 152 * ChainCfg<NB>::CTAS && (size_t)N * NB * sizeof(float) <= ChainCfg<NB>::MAX_VEC &&
         (cluster == 1 || chain_rounds<NB>(N) <= (NB < 32 ? 12 : 11));
}

struct ChainItem {
  int q, pl, pr;
  bool elim;
};
__device__ __forceinline__ int chain_fwd_tasks(int N, int Lc, int lvl) {
  return lvl == Lc ? 1 : lvl == 0 ? N / 2 : ((N - 1) >> lvl) + 1;
}
__device__ __forceinline__ ChainItem chain_fwd_item(int N, int Lc, int lvl, int t) {
  ChainItem w;
  const bool last = lvl == Lc;
  if (last) w.q = N;
  else if (lvl == 0) w.q = 2 * t + 1;
  else w.q = t < ((N - 1) >> lvl) ? (t + 1) << lvl : N;
  w.elim = last || (w.q < N && ctz32(w.q) == lvl);
  w.pl = w.pr = 0;
  if (lvl >= 1) {
    const int h = 1 << (lvl - 1);
    if (w.q < N) {
      w.pl = w.q - h;
      if (w.q + h <= N - 1) w.pr = w.q + h;
    } else {
      const int mm = ((N - 1) >> (lvl - 1)) << (lvl - 1);
      if (ctz32(mm) == lvl - 1) w.pl = mm;
    }
  }
  return w;
}

// z - sum_k l[k] y[k], y in shared memory, k in increasing order.
template <int NB>
__device__ __forceinline__ float chain_dot(const float (&l)[NB], const float *y, float z) {
  if constexpr (NB % 4 == 0) {
    const float4 *y4 = reinterpret_cast<const float4 *>(y);
#pragma unroll
    for (int g = 0; g < NB / 4; ++g) {
      const float4 v = y4[g];
      z = fmaf(-l[4 * g], v.x, z);
      z = fmaf(-l[4 * g + 1], v.y, z);
      z = fmaf(-l[4 * g + 2], v.z, z);
      z = fmaf(-l[4 * g + 3], v.w, z);
    }
  } else {
#pragma unroll
    for (int k = 0; k < NB; ++k) z = fmaf(-l[k], y[k], z);
  }
  return z;
}
template <int NB>
__device__ __forceinline__ void load_col(float (&c)[NB], const float *__restrict__ p) {
#pragma unroll
  for (int k = 0; k < NB; ++k) c[k] = p[k * NB];
}

// Forward substitution of tail s (as fwd_tail). vec: N * NB floats of shared
// memory, the partial sums and then the results of each position; the
// results also go to m.y for the backward kernel.
template <int NB>
__device__ __forceinline__ void fwd_tail_chain(const MixedState &m, const double *__restrict__ rhs, int s, float *vec,
                                               float (*sY)[NB]) {
  constexpr int TS = ChainCfg<NB>::TS, TEAMS = ChainCfg<NB>::TEAMS, NB2 = NB * NB;
  const Team<TS> tm;
  const int N = m.N, Lc = m.Lc, i = tm.lane, ir = i < NB ? i : 0;
  const size_t sb = (size_t)s * N;
  const bool xmode = coupled(m);
  float X[NB], Y[NB], L[NB], inv = 0.0f;
  double zr = 0.0;
  auto load_x = [&](const ChainItem &w) {
    if (w.pl) load_row<NB>(X, m.Lr + (sb + (N - w.pl)) * NB2 + ir * NB);
  };
  auto load_y = [&](const ChainItem &w) {
    if (w.pr) load_row<NB>(Y, m.Ll + (sb + (N - w.pr)) * NB2 + ir * NB);
  };
  auto load_l = [&](const ChainItem &w) {
    if (w.elim) {
      load_row<NB>(L, m.Ld + (sb + (N - w.q)) * NB2 + ir * NB);
      inv = m.invd[(sb + (N - w.q)) * NB + ir];
    }
  };
  auto load_r = [&](const ChainItem &w, int lvl) {
    if (lvl <= 1) zr = rhs[(sb + (N - w.q)) * NB + ir];
  };
  // the team's next position: at (lvl, t) or in a later level; false: none
  auto seek = [&](int &lvl, int &t) {
    while (lvl <= Lc && t >= chain_fwd_tasks(N, Lc, lvl)) {
      ++lvl;
      t = tm.id;
    }
    return lvl <= Lc;
  };
  int nl = 0, nt = tm.id;
  ChainItem w{};
  bool have = seek(nl, nt);
  if (have) {
    w = chain_fwd_item(N, Lc, nl, nt);
    load_r(w, nl);
    load_x(w);
    load_y(w);
    load_l(w);
  }
  for (int lvl = 0; lvl <= Lc; ++lvl) {
    const bool lastlvl = lvl == Lc;
    while (have && nl == lvl) {
      const ChainItem c = w;
      float *vq = vec + (N - c.q) * NB;
      float z = lvl <= 1 ? __double2float_rn(zr) : vq[ir];
      nt += TEAMS;
      have = seek(nl, nt);
      ChainItem n{};
      if (have) {
        n = chain_fwd_item(N, Lc, nl, nt);
        load_r(n, nl);
      }
      if (c.pl) z = chain_dot<NB>(X, vec + (N - c.pl) * NB, z);
      if (have) load_x(n);
      if (c.pr) z = chain_dot<NB>(Y, vec + (N - c.pr) * NB, z);
      if (have) load_y(n);
      if (c.elim) {
        if (TS <= 32) {
          const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            if (i == j) z *= inv;
            const float yj = __shfl_sync(tm.mask, z, base + j);
            if (i > j && i < NB) z = fmaf(-L[j], yj, z);
          }
        } else {
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            if (i == j) {
              z *= inv;
              sY[tm.id][j] = z;
            }
            tm.sync();
            if (i > j && i < NB) z = fmaf(-L[j], sY[tm.id][j], z);
          }
        }
        if (i < NB) m.y[(sb + (N - c.q)) * NB + i] = z;
      }
      // (lanes beyond NB repeat row 0)
      if (i < NB) vq[i] = z;
      if (have) load_l(n);
      w = n;
    }
    __syncthreads();
    if (lastlvl && !xmode) {
      // t_i = F_{i,1} y_1
      const int nr = m.nr;
      const double *Fs = m.F + (size_t)s * nr * NB;
      const float *y1 = vec;   // stage 1 (position N)
      for (int c = threadIdx.x; c < nr; c += blockDim.x) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < NB; ++k) acc = fma(Fs[c * NB + k], f2d_exact(y1[k]), acc);
        m.tb[(size_t)s * nr + c] = acc;
      }
    }
  }
}

// Backward substitution fused with x += d (as bwd_tail). vec: the
// corrections of the positions done so far.
template <int NB>
__device__ __forceinline__ void bwd_tail_chain(const MixedState &m, double *x, int iter, int s, float *vec,
                                               float (*sX)[NB]) {
  constexpr int TS = ChainCfg<NB>::TS, TEAMS = ChainCfg<NB>::TEAMS, NB2 = NB * NB;
  const Team<TS> tm;
  const int N = m.N, Lc = m.Lc, nr = m.nr, i = tm.lane, ir = i < NB ? i : 0;
  const size_t sb = (size_t)s * N;
  const bool xmode = coupled(m);
  __shared__ float sdh[64], sdl[64];   // d_0 as hi + lo floats (refined coupling columns)
  float B[NB], A[NB], L[NB], inv = 0.0f, yv = 0.0f;
  double xold = 0.0;
  auto tasks = [&](int lvl) { return lvl == Lc ? 1 : (((N - 1) >> lvl) + 1) / 2; };
  auto pos = [&](int lvl, int t) { return lvl == Lc ? N : (2 * t + 1) << lvl; };
  auto load_b = [&](int lvl, int q) {
    if (lvl < Lc) load_col<NB>(B, m.Lr + (sb + (N - q)) * NB2 + ir);
  };
  auto load_a = [&](int lvl, int q) {
    if (lvl < Lc && q > (1 << lvl)) load_col<NB>(A, m.Ll + (sb + (N - q)) * NB2 + ir);
  };
  auto load_l = [&](int q) {
    load_col<NB>(L, m.Ld + (sb + (N - q)) * NB2 + ir);
    inv = m.invd[(sb + (N - q)) * NB + ir];
  };
  auto load_v = [&](int q) {
    const size_t o = (sb + (N - q)) * NB + ir;
    yv = m.y[o];
    if (iter != 0) xold = x[o];
  };
  auto seek = [&](int &lvl, int &t) {
    while (lvl >= 0 && t >= tasks(lvl)) {
      --lvl;
      t = tm.id;
    }
    return lvl >= 0;
  };
  int nl = Lc, nt = tm.id;
  bool have = seek(nl, nt);
  int q = have ? pos(nl, nt) : 0;
  if (have) {
    load_v(q);
    load_b(nl, q);
    load_a(nl, q);
    load_l(q);
  }
  if (xmode) {
    for (int c = threadIdx.x; c < nr; c += blockDim.x) ff::split_d(__ldcg(m.d0 + c), sdh[c], sdl[c]);
    __syncthreads();
  }
  for (int lvl = Lc; lvl >= 0; --lvl) {
    while (have && nl == lvl) {
      const int cq = q;
      const size_t zoff = (sb + (N - cq)) * NB;
      float z = yv;
      const double xo = xold;
      nt += TEAMS;
      have = seek(nl, nt);
      q = have ? pos(nl, nt) : 0;
      if (have) load_v(q);
      if (lvl == Lc) {
        if (!xmode && i < NB) {
          double zd = f2d_exact(z);
          const double *Fs = m.F + (size_t)s * nr * NB;
          for (int c = 0; c < nr; ++c) zd = fma(-Fs[c * NB + i], __ldcg(m.d0 + c), zd);
          z = __double2float_rn(zd);
        }
        if (have) {
          load_b(nl, q);
          load_a(nl, q);
        }
      } else {
        const int h = 1 << lvl;
        const int a = cq - h, b = (cq + h <= N - 1) ? cq + h : N;
        z = chain_dot<NB>(B, vec + (N - b) * NB, z);
        if (have) load_b(nl, q);
        if (cq > h) z = chain_dot<NB>(A, vec + (N - a) * NB, z);
        if (have) load_a(nl, q);
      }
      if (TS <= 32) {
        const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
        for (int j = NB - 1; j >= 0; --j) {
          if (i == j) z *= inv;
          const float xj = __shfl_sync(tm.mask, z, base + j);
          if (i < j) z = fmaf(-L[j], xj, z);
        }
      } else {
#pragma unroll
        for (int j = NB - 1; j >= 0; --j) {
          if (i == j) {
            z *= inv;
            sX[tm.id][j] = z;
          }
          tm.sync();
          if (i < j) z = fmaf(-L[j], sX[tm.id][j], z);
        }
      }
      if (i < NB) {
        vec[(N - cq) * NB + i] = z;
        m.y[zoff + i] = z;
        double dz;
        if (xmode) {
          // d_i = z - X_i d_0 on this row, the product summed by Dot2
          const float *xr = m.Xc + (zoff + i) * m.ldc;
          float h = 0.0f, l = 0.0f;
          for (int c = 0; c < nr; ++c) ff::dot2_step_split(h, l, sdh[c], sdl[c], __ldcg(xr + c));
          float dh, e;
          ff::two_sum(z, -h, dh, e);
          dz = ff::to_double(dh, __fsub_rn(e, l));
        } else {
          dz = f2d_exact(z);
        }
        const double xv = iter == 0 ? dz : xo + dz;
        x[zoff + i] = xv;
        if (m.ffres) {
          float h, l;
          ff::split_d(xv, h, l);
          m.xh[zoff + i] = h;
          m.xl[zoff + i] = l;
          if (ff::out_of_range(xv)) m.status->ffbad = 1;
        }
      }
      if (have) load_l(q);
    }
    __syncthreads();
  }
}

}  // namespace mx
}  // namespace bm
