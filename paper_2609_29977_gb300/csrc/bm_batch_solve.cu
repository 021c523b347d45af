// Batched refinement-step kernels: one CTA per tail of every system
// (forward substitution with each system's root step in its last CTA,
// backward substitution with x += d, FP64 residual with each system's
// stopping test in its last CTA). See bm_batch.cu.
#include "bm_batch.cuh"

namespace bm {
namespace {
using namespace mx;

// Per-solve reset of the control blocks.
__global__ void k_batch_reset(BInst *inst, int ninst) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= ninst) return;
  IRCtl *c = inst[b].m.ctl;
  c->converged = 0;
  c->iters = 0;
  c->wmax = 0u;
  c->omega_prev = 0.0;
  inst[b].m.tickets[2] = 0u;
  inst[b].m.tickets[3] = 0u;
}

constexpr int kSubFloats = SubCfg<48>::floats(256);   // the widest block's

__global__ void __launch_bounds__(256, 3) k_batch_fwd(const BInst *inst, const BTail *tails, const double *const *rp,
                                                   double *const *xp, int iter) {
  // the tail's part, then the root step
  __shared__ __align__(16) double sbuf[kSubFloats / 2 > 64 * 64 + 128 ? kSubFloats / 2 : 64 * 64 + 128];
  const BTail t = tails[blockIdx.x];
  const BInst &I = inst[t.inst];
  pdl_wait();
  if (ir_done(I.m.ctl)) return;
  const double *rhs = iter == 0 ? rp[t.inst] : I.m.rho;
  switch (I.nb) {
#define X(n)                                                              \
  case n:                                                                 \
    fwd_tail<n>(I.m, rhs, t.s, 0, 1, (float *)sbuf);                       \
    if (last_cta(&I.m.tickets[2], (unsigned)I.S)) root_step<n>(I.m, rhs, xp[t.inst], iter, sbuf, I.S); \
    break;
    BM_BATCH_NB_LIST(X)
#undef X
  }
}

// Wide blocks keep the teams of two warps here: the CTA's registers are set
// by all block sizes (80 for three CTAs per SM), too few for the pair form's
// loads in flight. Batch of 16 systems, per pass: 179 us, pair form 284 us
// (262 us with two CTAs per SM). The forward form reads L_qq from shared
// memory and gains: 290 -> 240 us.
__global__ void __launch_bounds__(256, 3) k_batch_bwd(const BInst *inst, const BTail *tails, double *const *xp,
                                                   int iter) {
  __shared__ __align__(16) float sbuf[256];
  const BTail t = tails[blockIdx.x];
  const BInst &I = inst[t.inst];
  pdl_wait();
  if (ir_done(I.m.ctl)) return;
  switch (I.nb) {
#define X(n)                                                                           \
  case n:                                                                              \
    bwd_tail<n, false>(I.m, xp[t.inst], iter, t.s, 0, 1, sbuf);                        \
    break;
    BM_BATCH_NB_LIST(X)
#undef X
  }
}

// MINB: CTAs per SM, three (80 registers), or four (64, some spilling) where
// the large tails (large: those with at least half of the largest one's
// work) then run in fewer waves. 16 systems of 30 tails, N = 60, solve, us,
// three -> four: nb = 6 478 -> 464, 12 740 -> 710, 24 1417 -> 1320, 48 3987 -> 3641;
// with as many waves (8 systems of 100 tails, N = 100) 24 2809 -> 3015, 48
// 7504 -> 8321. By the number of all tails, a batch of 16 uneven systems took 5581 us
// for factor and solve instead of 5344.
inline bool four_ctas(long ctas) { return (ctas + 4 * 152 - 1) / (4 * 152) < (ctas + 3 * 152 - 1) / (3 * 152); }

template <int MINB>
__global__ void __launch_bounds__(256, MINB) k_batch_res(const BInst *inst, const BTail *tails, const double *const *rp,
                                                      double *const *xp, int iter, int max_iter, double tol) {
  __shared__ double sbuf[8 * ResCfg<48>::WARP];
  const BTail t = tails[blockIdx.x];
  const BInst &I = inst[t.inst];
  pdl_wait();
  if (ir_done(I.m.ctl)) return;
  const double *r = rp[t.inst];
  const double *x = xp[t.inst];
  switch (I.nb) {
#define X(n)                                     \
  case n:                                        \
    residual_tail<n>(I.m, r, x, t.s, sbuf);      \
    break;
    BM_BATCH_NB_LIST(X)
#undef X
  }
  if (last_cta(&I.m.tickets[3], (unsigned)I.S)) residual_finish(I.m, r, x, I.nb, iter, max_iter, tol);
}

}  // namespace

void batch_launch_reset(BInst *inst, int ninst, cudaStream_t st) {
  k_batch_reset<<<(ninst + 127) / 128, 128, 0, st>>>(inst, ninst);
}

void batch_launch_solve_iteration(const BInst *inst, const BTail *tails, int ntails, int large,
                                  const double *const *r, double *const *x, int iter, int max_iter, double tol,
                                  cudaStream_t st) {
  launch_pdl(k_batch_fwd, (unsigned)ntails, 256, 0, st, inst, tails, r, x, iter);
  launch_pdl(k_batch_bwd, (unsigned)ntails, 256, 0, st, inst, tails, x, iter);
  launch_pdl(four_ctas(large) ? k_batch_res<4> : k_batch_res<3>, (unsigned)ntails, 256, 0, st, inst, tails, r, x, iter,
             max_iter, tol);
}

}  // namespace bm
