// FP64 triangular solves (Alg. 2) with one thread-block cluster per tail.
//
// The forward substitution of a tail walks the odd-even levels of
// Gamma_{N-1} upwards and its backward substitution walks them downwards
// (Sec. IV-C); all levels of one tail run inside one launch, the CTAs of
// the tail's cluster splitting the positions of each level and meeting at a
// cluster barrier between levels. Each position is handled by a team of TS
// lanes, one lane per block row: the row's gather of the neighbours'
// contributions is one dependent FMA chain, and the triangular solve with
// the diagonal block passes each new component to the other rows with a
// warp shuffle (through shared memory for teams wider than a warp).
// Values written by other CTAs of the cluster are read with L2-only loads
// after the barrier (release/acquire at cluster scope).
//
// Three launches per solve: tail forward (+ x_1 forward and F_{i,1} y_1),
// the root step (bm_fp64.cu), tail backward (root propagation, x_1, levels).
#include "bm_team.cuh"

namespace bm {
namespace {

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

template <int NB>
struct SolveCfg {
  static constexpr int TS = NB <= 4 ? 4 : NB <= 8 ? 8 : NB <= 16 ? 16 : NB <= 32 ? 32 : 64;
  static constexpr int THREADS = 256;
  static constexpr int TEAMS = THREADS / TS;
  // CTAs per SM that the register-capped instantiation must allow: with
  // one CTA per tail, four per SM keep up to 608 tails in a single wave on
  // 152 SMs (the uncapped one, 80 registers at nb = 24, fits three)
  static constexpr int MINB = NB <= 32 ? 4 : 2;
};

// Whether a launch of S * CS CTAs needs the register-capped kernels: more
// CTAs than three per SM would otherwise run in a second, mostly empty wave.
inline bool solve_capped(int S, int CS) { return (long)S * CS > 3 * 152; }

// Forward levels of one tail, then x_1: y_1 = L_{i,1}^{-1} z_1 and
// t_i = F_{i,1} y_1. Grid: S * CS CTAs, clusters of CS.
template <int NB, int MINB>
__global__ void __launch_bounds__(256, MINB) k_solve_fwd_tail(F64View v, const double *__restrict__ r, int CS) {
  constexpr int TS = SolveCfg<NB>::TS, TEAMS = SolveCfg<NB>::TEAMS, NB2 = NB * NB;
  __shared__ double sY[TEAMS][NB];
  const Team<TS> tm;
  const int crank = (int)cluster_rank();
  const int s = blockIdx.x / CS;
  const int N = v.N, Lc = v.Lc;
  const size_t sb = (size_t)s * N;
  const int i = tm.lane;   // block row handled by this lane (if < NB)
  pdl_wait();
  for (int lvl = 0; lvl <= Lc; ++lvl) {
    const bool last = lvl == Lc;   // x_1
    const int ntask = last ? 1 : (lvl == 0 ? N / 2 : ((N - 1) >> lvl) + 1);
    for (int t = crank * TEAMS + tm.id; t < ntask; t += CS * TEAMS) {
      int q;
      if (last) q = N;
      else if (lvl == 0) q = 2 * t + 1;
      else {
        const int cnt = (N - 1) >> lvl;
        q = t < cnt ? (t + 1) << lvl : N;
      }
      const bool elim = last || (q < N && ctz32(q) == lvl);
      const size_t zoff = (sb + (N - q)) * NB;
      double z = 0.0;
      if (i < NB) {
        z = (lvl <= 1) ? r[zoff + i] : __ldcg(v.zt + zoff + i);
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
            const double *L = v.Lr + (sb + (N - pl)) * NB2 + i * NB;
            const double *y = v.y + (sb + (N - pl)) * NB;
#pragma unroll
            for (int k = 0; k < NB; ++k) z = fma(-L[k], __ldcg(y + k), z);
          }
          if (pr) {
            const double *L = v.Ll + (sb + (N - pr)) * NB2 + i * NB;
            const double *y = v.y + (sb + (N - pr)) * NB;
#pragma unroll
            for (int k = 0; k < NB; ++k) z = fma(-L[k], __ldcg(y + k), z);
          }
        }
      }
      if (!elim) {
        if (i < NB) v.zt[zoff + i] = z;
        continue;
      }
      // y = L_qq^{-1} z as M w = z, y = inv .* w with the unit lower
      // factor M = L_qq diag(L_qq)^-1, whose row i is column i of the
      // stored block's upper triangle (read coalesced across the lanes)
      const double *Mrow = v.Ld + (sb + (N - q)) * NB2 + (i < NB ? i : 0);
      const double inv = i < NB ? v.invd[zoff + i] : 0.0;
      if (TS <= 32) {
        const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
        for (int j = 0; j < NB - 1; ++j) {
          const double wj = __shfl_sync(tm.mask, z, base + j);
          if (i > j && i < NB) z = fma(-Mrow[j * NB], wj, z);
        }
        z *= inv;
        if (i < NB) sY[tm.id][i] = z;
        tm.sync();
      } else {
#pragma unroll
        for (int j = 0; j < NB - 1; ++j) {
          if (i == j) sY[tm.id][j] = z;
          tm.sync();
          if (i > j && i < NB) z = fma(-Mrow[j * NB], sY[tm.id][j], z);
        }
        z *= inv;
        tm.sync();
        if (i < NB) sY[tm.id][i] = z;
      }
      if (i < NB) v.y[zoff + i] = z;
      if (last) {
        tm.sync();
        const int nr = v.nr;
        const double *Fs = v.F + (size_t)s * nr * NB;
        for (int c = i; c < nr; c += TS) {
          double acc = 0.0;
#pragma unroll
          for (int k = 0; k < NB; ++k) acc = fma(Fs[c * NB + k], sY[tm.id][k], acc);
          v.tb[(size_t)s * nr + c] = acc;
        }
      }
      tm.sync();
    }
    cluster_sync();
  }
}

// Backward: root propagation y_1 -= F_{i,1}^T x_0, x_1 = L_{i,1}^{-T} y_1,
// then levels Lc-1..0: x_q = L_qq^{-T}(y_q - L_{a,q}^T x_a - L_{b,q}^T x_b),
// written in natural order.
template <int NB, int MINB>
__global__ void __launch_bounds__(256, MINB) k_solve_bwd_tail(F64View v, double *__restrict__ x, int CS) {
  constexpr int TS = SolveCfg<NB>::TS, TEAMS = SolveCfg<NB>::TEAMS, NB2 = NB * NB;
  __shared__ double sX[TEAMS][NB];
  const Team<TS> tm;
  const int crank = (int)cluster_rank();
  const int s = blockIdx.x / CS;
  const int N = v.N, Lc = v.Lc, nr = v.nr;
  const size_t sb = (size_t)s * N;
  const size_t n0 = (size_t)v.S * N * NB;
  const int i = tm.lane;
  pdl_wait();
  for (int lvl = Lc; lvl >= 0; --lvl) {
    const bool first = lvl == Lc;   // x_1
    const int ntask = first ? 1 : (((N - 1) >> lvl) + 1) / 2;
    for (int t = crank * TEAMS + tm.id; t < ntask; t += CS * TEAMS) {
      const int q = first ? N : (2 * t + 1) << lvl;
      const size_t zoff = (sb + (N - q)) * NB;
      double z = 0.0;
      if (i < NB) {
        z = v.y[zoff + i];
        if (first) {
          const double *Fs = v.F + (size_t)s * nr * NB;
          for (int c = 0; c < nr; ++c) z = fma(-Fs[c * NB + i], __ldcg(x + n0 + c), z);
        } else {
          const int h = 1 << lvl;
          const int a = q - h, b = (q + h <= N - 1) ? q + h : N;
          const double *Lb = v.Lr + (sb + (N - q)) * NB2 + i;
          const double *xb = x + (sb + (N - b)) * NB;
#pragma unroll
          for (int k = 0; k < NB; ++k) z = fma(-Lb[k * NB], __ldcg(xb + k), z);
          if (q > h) {
            const double *La = v.Ll + (sb + (N - q)) * NB2 + i;
            const double *xa = x + (sb + (N - a)) * NB;
#pragma unroll
            for (int k = 0; k < NB; ++k) z = fma(-La[k * NB], __ldcg(xa + k), z);
          }
        }
      }
      // x = L_qq^{-T} z as M^T x = inv .* z with the unit lower factor
      // M = L_qq diag(L_qq)^-1, whose column i is row i of the stored
      // block's upper triangle
      double Mcol[NB];
      const double *Ld = v.Ld + (sb + (N - q)) * NB2 + (i < NB ? i : 0) * NB;
#pragma unroll
      for (int k = 0; k < NB; ++k) Mcol[k] = Ld[k];
      const double inv = i < NB ? v.invd[zoff + i] : 0.0;
      z *= inv;
      if (TS <= 32) {
        const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
        for (int j = NB - 1; j > 0; --j) {
          const double xj = __shfl_sync(tm.mask, z, base + j);
          if (i < j) z = fma(-Mcol[j], xj, z);
        }
      } else {
#pragma unroll
        for (int j = NB - 1; j > 0; --j) {
          if (i == j) sX[tm.id][j] = z;
          tm.sync();
          if (i < j) z = fma(-Mcol[j], sX[tm.id][j], z);
        }
      }
      if (i < NB) x[zoff + i] = z;
      tm.sync();
    }
    cluster_sync();
  }
}

// The same substitutions for few tails: one CTA per tail, its vectors in
// shared memory, the factor's rows one position ahead in registers. With few
// tails a level costs a trip to L2 for the neighbours' vectors, one to memory
// for the factor's rows and a cluster barrier on top of its arithmetic; here
// the vectors stay on the SM and a team's next rows, which do not depend on
// the substitution, are requested as soon as the registers of the present
// ones are free, across the barrier between levels. Same operations per row
// in the same order. Solve, clusters -> this form, us: S = 4, N = 16, nb = 4
// 22.6 -> 18.5; S = 37, N = 50, nb = 12 57 -> 45; S = N = 64, nb = 12 51 -> 49;
// S = 100, N = 160, nb = 16 164 -> 152; S = 150, N = 128, nb = 24 277 -> 228.
// The FP64 pipe (64 cycles per instruction) is what is left.
template <int NB>
struct ChainCfg {
  static constexpr bool ON = NB <= 24;               // three rows per lane in registers
  static constexpr int CTAS = NB <= 16 ? 2 : 1;      // per SM
  static constexpr size_t MAX_VEC = 96 * 1024;       // bytes of one tail's vectors
};

// Positions that a team walks one after another over all levels.
template <int NB>
int chain_rounds(int N) {
  const int Lc = chain_levels(N), T = SolveCfg<NB>::TEAMS;
  int r = 1;
  for (int l = 0; l < Lc; ++l) r += ((l == 0 ? N / 2 : ((N - 1) >> l) + 1) + T - 1) / T;
  return r;
}
// One wave of CTAs, and either the other form has one CTA per tail as well
// or a team has few positions to walk, so that a cluster's further teams save
// less than its barriers cost: with more rounds (S, N, nb; rounds, cluster size)
// 8, 64, 24 (15, 8): 89 -> 121 us; 20, 200, 12 (24, 4): 71 -> 113;
// 60, 100, 24 (23, 2): 146 -> 186; with at most twelve none is slower.
template <int NB>
bool chain_applies(int S, int N, int cluster) {
  return ChainCfg<NB>::ON && S <= 152 * ChainCfg<NB>::CTAS &&
         (size_t)N * NB * sizeof(double) <= ChainCfg<NB>::MAX_VEC && (cluster == 1 || chain_rounds<NB>(N) <= 12);
}

template <int NB>
__device__ __forceinline__ double chain_dot(const double (&l)[NB], const double *y, double z) {
#pragma unroll
  for (int k = 0; k < NB; ++k) z = fma(-l[k], y[k], z);
  return z;
}

template <int NB>
__global__ void __launch_bounds__(256, ChainCfg<NB>::CTAS) k_solve_fwd_chain(F64View v, const double *__restrict__ r) {
  constexpr int TS = SolveCfg<NB>::TS, TEAMS = SolveCfg<NB>::TEAMS, NB2 = NB * NB;
  extern __shared__ __align__(16) double vec[];   // partial sums, then results, by natural stage
  const Team<TS> tm;
  const int N = v.N, Lc = v.Lc, s = blockIdx.x, i = tm.lane, ir = i < NB ? i : 0;
  const size_t sb = (size_t)s * N;
  double X[NB], Y[NB], M[NB], inv = 0.0, zr = 0.0;
  auto tasks = [&](int lvl) { return lvl == Lc ? 1 : lvl == 0 ? N / 2 : ((N - 1) >> lvl) + 1; };
  struct Item {
    int q, pl, pr;
    bool elim;
  };
  auto item = [&](int lvl, int t) {
    Item w;
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
        const int m = ((N - 1) >> (lvl - 1)) << (lvl - 1);
        if (ctz32(m) == lvl - 1) w.pl = m;
      }
    }
    return w;
  };
  auto load_x = [&](const Item &w) {
    const double *p = v.Lr + (sb + (N - w.pl)) * NB2 + ir * NB;
    if (w.pl)
#pragma unroll
      for (int k = 0; k < NB; ++k) X[k] = p[k];
  };
  auto load_y = [&](const Item &w) {
    const double *p = v.Ll + (sb + (N - w.pr)) * NB2 + ir * NB;
    if (w.pr)
#pragma unroll
      for (int k = 0; k < NB; ++k) Y[k] = p[k];
  };
  auto load_m = [&](const Item &w) {   // row i of the unit factor: column i of the block's upper triangle
    const double *p = v.Ld + (sb + (N - w.q)) * NB2 + ir;
    if (w.elim) {
#pragma unroll
      for (int j = 0; j < NB - 1; ++j) M[j] = p[j * NB];
      inv = v.invd[(sb + (N - w.q)) * NB + ir];
    }
  };
  auto load_r = [&](const Item &w, int lvl) {
    if (lvl <= 1) zr = r[(sb + (N - w.q)) * NB + ir];
  };
  auto seek = [&](int &lvl, int &t) {
    while (lvl <= Lc && t >= tasks(lvl)) {
      ++lvl;
      t = tm.id;
    }
    return lvl <= Lc;
  };
  pdl_wait();
  int nl = 0, nt = tm.id;
  Item w{};
  bool have = seek(nl, nt);
  if (have) {
    w = item(nl, nt);
    load_r(w, nl);
    load_x(w);
    load_y(w);
    load_m(w);
  }
  for (int lvl = 0; lvl <= Lc; ++lvl) {
    while (have && nl == lvl) {
      const Item c = w;
      double *vq = vec + (N - c.q) * NB;
      double z = lvl <= 1 ? zr : vq[ir];
      nt += TEAMS;
      have = seek(nl, nt);
      Item n{};
      if (have) {
        n = item(nl, nt);
        load_r(n, nl);
      }
      if (c.pl) z = chain_dot<NB>(X, vec + (N - c.pl) * NB, z);
      if (have) load_x(n);
      if (c.pr) z = chain_dot<NB>(Y, vec + (N - c.pr) * NB, z);
      if (have) load_y(n);
      if (c.elim) {
        const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
        for (int j = 0; j < NB - 1; ++j) {
          const double wj = __shfl_sync(tm.mask, z, base + j);
          if (i > j && i < NB) z = fma(-M[j], wj, z);
        }
        z *= inv;
        if (i < NB) v.y[(sb + (N - c.q)) * NB + i] = z;
      }
      if (i < NB) vq[i] = z;
      if (have) load_m(n);
      w = n;
    }
    __syncthreads();
  }
  const int nr = v.nr;   // t_i = F_{i,1} y_1 (stage 1 is the first of vec)
  const double *Fs = v.F + (size_t)s * nr * NB;
  for (int c = threadIdx.x; c < nr; c += blockDim.x) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) acc = fma(Fs[c * NB + k], vec[k], acc);
    v.tb[(size_t)s * nr + c] = acc;
  }
}

template <int NB>
__global__ void __launch_bounds__(256, ChainCfg<NB>::CTAS) k_solve_bwd_chain(F64View v, double *__restrict__ x) {
  constexpr int TS = SolveCfg<NB>::TS, TEAMS = SolveCfg<NB>::TEAMS, NB2 = NB * NB;
  extern __shared__ __align__(16) double vec[];   // x of the positions done so far, by natural stage
  const Team<TS> tm;
  const int N = v.N, Lc = v.Lc, nr = v.nr, s = blockIdx.x, i = tm.lane, ir = i < NB ? i : 0;
  const size_t sb = (size_t)s * N, n0 = (size_t)v.S * N * NB;
  double B[NB], A[NB], M[NB], inv = 0.0, yv = 0.0;
  auto tasks = [&](int lvl) { return lvl == Lc ? 1 : (((N - 1) >> lvl) + 1) / 2; };
  auto pos = [&](int lvl, int t) { return lvl == Lc ? N : (2 * t + 1) << lvl; };
  auto load_b = [&](int lvl, int q) {
    const double *p = v.Lr + (sb + (N - q)) * NB2 + ir;
    if (lvl < Lc)
#pragma unroll
      for (int k = 0; k < NB; ++k) B[k] = p[k * NB];
  };
  auto load_a = [&](int lvl, int q) {
    const double *p = v.Ll + (sb + (N - q)) * NB2 + ir;
    if (lvl < Lc && q > (1 << lvl))
#pragma unroll
      for (int k = 0; k < NB; ++k) A[k] = p[k * NB];
  };
  auto load_m = [&](int q) {   // column i of the unit factor: row i of the block's upper triangle
    const double *p = v.Ld + (sb + (N - q)) * NB2 + ir * NB;
#pragma unroll
    for (int k = 1; k < NB; ++k) M[k] = p[k];
    inv = v.invd[(sb + (N - q)) * NB + ir];
  };
  auto load_v = [&](int q) { yv = v.y[(sb + (N - q)) * NB + ir]; };
  auto seek = [&](int &lvl, int &t) {
    while (lvl >= 0 && t >= tasks(lvl)) {
      --lvl;
      t = tm.id;
    }
    return lvl >= 0;
  };
  pdl_wait();
  int nl = Lc, nt = tm.id;
  bool have = seek(nl, nt);
  int q = have ? pos(nl, nt) : 0;
  if (have) {
    load_v(q);
    load_b(nl, q);
    load_a(nl, q);
    load_m(q);
  }
  for (int lvl = Lc; lvl >= 0; --lvl) {
    while (have && nl == lvl) {
      const int cq = q;
      double z = yv;
      nt += TEAMS;
      have = seek(nl, nt);
      q = have ? pos(nl, nt) : 0;
      if (have) load_v(q);
      if (lvl == Lc) {
        const double *Fs = v.F + (size_t)s * nr * NB;
        for (int c = 0; c < nr; ++c) z = fma(-Fs[c * NB + ir], __ldcg(x + n0 + c), z);
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
      z *= inv;
      const int base = (threadIdx.x & 31) & ~(TS - 1);
#pragma unroll
      for (int j = NB - 1; j > 0; --j) {
        const double xj = __shfl_sync(tm.mask, z, base + j);
        if (i < j) z = fma(-M[j], xj, z);
      }
      if (i < NB) {
        vec[(N - cq) * NB + i] = z;
        x[(sb + (N - cq)) * NB + i] = z;
      }
      if (have) load_m(q);
    }
    __syncthreads();
  }
}

int pick_cluster(int S) {
  int cs = 1;
  while (cs < 8 && S * cs * 2 <= 152) cs <<= 1;
  return cs;
}

template <int NB>
cudaError_t launch_tail_kernel(void (*kern)(F64View, const double *, int), const F64View &v, const double *r,
                               cudaStream_t st) {
  const int CS = pick_cluster(v.S);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(v.S * CS));
  cfg.blockDim = dim3(SolveCfg<NB>::THREADS);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, v, r, CS);
}

template <int NB>
cudaError_t launch_bwd_kernel(const F64View &v, double *x, cudaStream_t st) {
  const int CS = pick_cluster(v.S);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(v.S * CS));
  cfg.blockDim = dim3(SolveCfg<NB>::THREADS);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (solve_capped(v.S, CS)) return cudaLaunchKernelEx(&cfg, k_solve_bwd_tail<NB, SolveCfg<NB>::MINB>, v, x, CS);
  return cudaLaunchKernelEx(&cfg, k_solve_bwd_tail<NB, 1>, v, x, CS);
}

template <int NB>
bool launch_chain(const F64View &v, const double *r, double *x, cudaStream_t st);

}  // namespace

void f64_launch_solve_root(const F64View &v, const double *r, double *x, cudaStream_t st);

namespace {
// The solve in the form for few tails, where it applies.
template <int NB>
bool launch_chain(const F64View &v, const double *r, double *x, cudaStream_t st) {
  if constexpr (ChainCfg<NB>::ON) {
    if (!chain_applies<NB>(v.S, v.N, pick_cluster(v.S))) return false;
    const size_t vec = (size_t)v.N * NB * sizeof(double);
    launch_pdl(k_solve_fwd_chain<NB>, (unsigned)v.S, 256, vec, st, v, r);
    f64_launch_solve_root(v, r, x, st);
    launch_pdl(k_solve_bwd_chain<NB>, (unsigned)v.S, 256, vec, st, v, x);
    return true;
  }
  return false;
}

template <int NB>
cudaError_t prepare_chain() {
  if constexpr (ChainCfg<NB>::ON) {
    const cudaError_t e = cudaFuncSetAttribute(k_solve_fwd_chain<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)ChainCfg<NB>::MAX_VEC);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_solve_bwd_chain<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)ChainCfg<NB>::MAX_VEC);
  }
  return cudaSuccess;
}
}  // namespace

// The cluster solves substitute with the scaled unit factor that the
// compile-time tail factor stores above each diagonal block's diagonal, so
// they cover exactly the tail factor's block sizes.
#define BM_SOLVE_NB_LIST(X) BM_TAIL_NB_LIST(X)

bool f64_cluster_solve_supported(int nb) {
  switch (nb) {
#define X(n) case n:
    BM_SOLVE_NB_LIST(X)
#undef X
    return true;
  }
  return false;
}

// Shared-memory limits of the solve kernels, once per device.
cudaError_t f64_solve_prepare() {
  cudaError_t e = cudaSuccess;
#define X(n) \
  if (e == cudaSuccess) e = prepare_chain<n>();
  BM_SOLVE_NB_LIST(X)
#undef X
  return e;
}

void f64_cluster_launch_solve(const F64View &v, const double *r, double *x, cudaStream_t st) {
  switch (v.nb) {
#define X(n)                                                    \
  case n:                                                       \
    if (launch_chain<n>(v, r, x, st)) break;                    \
    launch_tail_kernel<n>(solve_capped(v.S, pick_cluster(v.S)) ? k_solve_fwd_tail<n, SolveCfg<n>::MINB> \
                                                               : k_solve_fwd_tail<n, 1>, v, r, st); \
    f64_launch_solve_root(v, r, x, st);                         \
    launch_bwd_kernel<n>(v, x, st);                             \
    break;
    BM_SOLVE_NB_LIST(X)
#undef X
  }
}

}  // namespace bm
