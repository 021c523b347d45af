// FP64 block products on the tensor cores, and the tail tasks built on them.
//
// GB300 retires one FP64 warp instruction per 64 cycles per SM sub-partition
// (DMMA shares that pipe and is no faster), so the block updates
// X X^T, A B^T of the tail factor are bound by the FP64 pipe. Here their
// products are formed exactly on the FP16 tensor cores instead (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 2012, with integer digits):
//
//   * a row x of an operand is read as fixed point relative to its largest
//     exponent E (|x_k| < 2^(E-1022)): q_k = x_k 2^62 / 2^(E-1022), truncated,
//     |q_k| < 2^62, and q_k = sum_i d_i 2^(9(6-i)) with seven digits d_i in
//     [-256, 256]. Adding 256 to every digit position first makes each digit
//     a plain bit field; the field and the removal of the 256 cost one FP16
//     addition for two digits.
//   * digit products d_i e_j are at most 2^16, so the sums over k of all
//     pairs with i + j = s are integers below 2^24 for k <= 32 (s + 1 pairs),
//     and FP32 accumulation in mma.sync (f16 operands) is exact. For nb = 48
//     only the sums of s = 5, 6 can exceed 2^24, and then by rounding a unit
//     that is 2^-61 of the largest product.
//   * the pairs with i + j <= 6 (28 products) are kept. Relative to X Y, the
//     powers of two above the largest entries of the two rows (up to twice
//     those entries each), a term k loses at most 6 2^16 2^45 / 2^124 = 2^-60.4
//     by the pairs left out and 2^-61 by the truncation of q, 2^-59.6 together,
//     a sum over K terms K times that at worst (2^-55 for K = 24, 2^-54 for 48).
//   * the seven sums are put together in 64-bit integers, at most two units
//     short by truncation (2^-57 of X Y for K <= 24, 2^-56 above), and turned
//     into a double by integer instructions, rounded to nearest, so a fill
//     block needs one FP64 multiplication (up_scale) and an update one FMA per
//     entry instead of nb (or 2 nb).
//
// Where each row carries one scale the loss stays within the backward error
// of an FMA chain, nb 2^-53 sqrt(K_ii K_jj): rows of L and of X do (|x_i| <=
// sqrt(K_ii), whatever the units of the variables), and the operands of the
// panels' inverses are brought to it (column_scale). Measured componentwise
// backward error of the solution, geometric mean over six generated systems
// whose variables have like units (before the columns were scaled, which moves
// solutions of such systems by rounding only), FMA chain -> sliced: 7.2e-16 ->
// 2.8e-16 (nb = 16), 6.8e-16 -> 2.7e-16 (24), 6.2e-16 -> 2.4e-16 (32), 5.7e-16
// -> 1.9e-16 (48). A row whose largest exponent is that of inf or NaN makes
// every product with it NaN, which a later pivot reports.
//
// What bounds the level kernels now (S = 128, N = 128, nb = 24, level 1, 242
// us, 255 before the register-resident trsm): nothing alone. Four warps per
// scheduler (14 KB of blocks each) issue in 45% of the cycles; ALU pipe 50%,
// FP64 pipe 32%, tensor pipe 26%. Tried and slower: the Cholesky in panels
// of eight columns on rows held by lanes (level 0 284 -> 301 us: its FP64
// instructions are the same, and fewer lanes of each do work), and substitution
// within the panels by FP64 FMAs instead of the inverted diagonal blocks
// (S = 512: 4047 against 3900 us for factor and solve).
#pragma once

#include "bm_team.cuh"

namespace bm {
namespace sliced {

constexpr int ND = 7;   // digits of 9 bits

// Block sizes whose FP64 tails use the sliced products (the line is drawn at
// Ops in bm_tail_factor.cuh).
template <typename T, int NB>
struct Use {
  static constexpr bool value = sizeof(T) == sizeof(double) && NB % 8 == 0 && NB >= 16;
};

// Bias that makes all seven digits non-negative: 256 at every digit.
constexpr unsigned long long kBias = 0x4020100804020100ull;   // sum_i 256 * 2^(9 i), i = 0..6

// x as fixed point relative to the biased exponent E of its row's largest
// entry, plus kBias.
__device__ __forceinline__ unsigned long long biased_fixed(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32) | (unsigned)__double2loint(x);
  const unsigned sh = min((unsigned)(E - (int)(e ? e : 1u)), 63u);   // (63 too for a row of zeros, whatever its E)
  const unsigned long long q = (m << 9) >> sh;
  return hi < 0 ? kBias - q : kBias + q;
}

// The digits of two neighbouring entries as FP16 pairs, most significant
// first (the operand registers of mma.sync m16n8k8/k16 hold two
// neighbouring k of one row), relative to the exponents E0 and E1.
__device__ __forceinline__ void digits(double x0, double x1, int E0, int E1, unsigned (&d)[ND]) {
  const unsigned long long a = biased_fixed(x0, E0), b = biased_fixed(x1, E1);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    const int sh = 9 * (ND - 1 - i);
    const unsigned ta = (unsigned)(a >> sh), tb = (unsigned)(b >> sh);
    // 0x6400 is the FP16 number 1024; its low bits count units
    const unsigned w = (__byte_perm(ta, tb, 0x5410) & (i == 0 ? 0x03ff03ffu : 0x01ff01ffu)) | 0x64006400u;
    unsigned r;
    asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0x65006500u));   // minus 1024 + 256
    d[i] = r;
  }
}

__device__ __forceinline__ void digits(double x0, double x1, int E, unsigned (&d)[ND]) { digits(x0, x1, E, E, d); }

__device__ __forceinline__ void mma_k16(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                        unsigned b0, unsigned b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&c)[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(b0));
}

// Eight rows x K columns of an operand as a lane holds them: entries (row
// lane/4, columns 8 g + 2 (lane%4) + {0, 1}), x[g]. That is the operand
// layout of mma.sync for A (rows) and for B (rows of B^T), and also the
// layout of the product's accumulators.
template <int K>
__device__ __forceinline__ void load_rows(double (&x)[K / 8][2], const double *__restrict__ base, int ld,
                                          int row, int nrows) {
  const int tig = threadIdx.x & 3;
#pragma unroll
  for (int g = 0; g < K / 8; ++g) {
    const int k = 8 * g + 2 * tig;
    double2 v = make_double2(0.0, 0.0);
    if (row < nrows) v = *reinterpret_cast<const double2 *>(base + row * ld + k);
    x[g][0] = v.x;
    x[g][1] = v.y;
  }
}

// Largest biased exponent of each row over x[0..KG), at least 1; kBadRow for
// a row with inf or NaN, which makes every product with it NaN (assemble).
constexpr int kBadRow = 1 << 20;
template <int KG, int KGX>
__device__ __forceinline__ int row_exponent(const double (&x)[KGX][2]) {
  unsigned mx = 0;
#pragma unroll
  for (int g = 0; g < KG; ++g)
    mx = max(mx, max((unsigned)__double2hiint(x[g][0]) & 0x7fffffffu, (unsigned)__double2hiint(x[g][1]) & 0x7fffffffu));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  const int E = (int)(mx >> 20);
  return E == 0x7ff ? kBadRow : max(E, 1);
}

// c[s] += the digit products with i + j = s of one group of 8 (or, with
// TWO, 16) columns; a0, a1: rows 0-7 and 8-15 of the tile, b: columns.
__device__ __forceinline__ void accumulate8(float (&c)[ND][4], const unsigned (&a0)[ND], const unsigned (&a1)[ND],
                                            const unsigned (&b)[ND]) {
#pragma unroll
  for (int j = 0; j < ND; ++j)
#pragma unroll
    for (int i = 0; i + j < ND; ++i) mma_k8(c[i + j], a0[i], a1[i], b[j]);
}
__device__ __forceinline__ void accumulate16(float (&c)[ND][4], const unsigned (&a0)[2][ND],
                                             const unsigned (&a1)[2][ND], const unsigned (&b)[2][ND]) {
#pragma unroll
  for (int j = 0; j < ND; ++j)
#pragma unroll
    for (int i = 0; i + j < ND; ++i)
      mma_k16(c[i + j], a0[0][i], a1[0][i], a0[1][i], a1[1][i], b[0][j], b[1][j]);
}

__device__ __forceinline__ void clear(float (&c)[ND][4]) {
#pragma unroll
  for (int s = 0; s < ND; ++s)
#pragma unroll
    for (int t = 0; t < 4; ++t) c[s][t] = 0.0f;
}

// The double nearest to (sum_s c_s 2^(9(12-s))) 2^-124 2^(Ea-1022) 2^(Eb-1022)
// after a truncation (of the sums of s = 5 and 6) by less than two units of V:
// 2^-57 (K <= 24) or 2^-56 of the two rows' powers of two. |c_s| as bounded above: the sum
// is below 2^(124 + log2 K), so the unit 2^66 (K <= 24) or 2^67 keeps the
// 64-bit integer in range.
template <int K>
__device__ __forceinline__ double assemble(const float (&c)[ND][4], int t, int Ea, int Eb) {
  constexpr int UP = K <= 24 ? 15 : 14;
  int v[ND];
#pragma unroll
  for (int s = 0; s < ND; ++s) v[s] = __float2int_rn(c[s][t]);
  long long V = (long long)((v[5] >> (18 - UP)) + (v[6] >> (27 - UP)));
  V += (long long)v[4] * (1 << (UP - 9));
  V += (long long)v[3] * (1 << UP);
  V += (long long)v[2] * (1 << (UP + 9));
  int hi = (int)(V >> 32) + v[1] * (1 << (UP + 18 - 32)) + v[0] * (1 << (UP + 27 - 32));
  unsigned lo = (unsigned)V;
  const int sg = hi >> 31;
  const unsigned long long a =
      (((unsigned long long)(unsigned)(hi ^ sg) << 32) | (lo ^ (unsigned)sg)) + (unsigned long long)(sg & 1);
  const int n = __clzll((long long)a);
  const unsigned long long m = a << n;                                  // leading one at bit 63
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);          // 2^52 <= r <= 2^53
  // a 2^(81-UP-124) = (m 2^-63) 2^(63-n) 2^(-43-UP); exponents Ea, Eb as 2^(E-1022)
  const int e = (63 - n) - 43 - UP + (Ea - 1022) + (Eb - 1022) + 1023;  // biased exponent of the result
  unsigned rh = (unsigned)(r >> 32) + ((unsigned)(e - 1) << 20), rl = (unsigned)r;
  if ((unsigned)(e - 1) >= 2046u || a == 0ull) {   // zero, underflow; overflow; inf or NaN in a row
    rl = 0u;
    rh = Ea == kBadRow || Eb == kBadRow ? 0x7ff80000u : a == 0ull || e < 1 ? 0u : 0x7ff00000u;
  }
  return __hiloint2double((int)(rh | ((unsigned)sg & 0x80000000u)), (int)rl);
}

// Products are put together 2^64 times too large and scaled back (f = 2^-64)
// by the FP64 instruction that takes them up, so that what is subnormal is
// rounded and not lost (K near the lower end of the range). Not for rows with
// entries from 2^448 on, where the scaled product could overflow: K_ii is
// above 2^896 there, and with any K_jj a product below 2^-1022 does not show.
// S = 512, N = 128, nb = 24: factor and solve 3836 -> 3862 us, nearly all of
// it in the updates of rows and the fill; S = 100, N = 160, nb = 16: 605 both.
__device__ __forceinline__ int up_scale(int E) { return E < 1023 + 448 ? 64 : 0; }
__device__ __forceinline__ double down_scale(int up) { return __hiloint2double((1023 - up) << 20, 0); }

// Calls out(i, j, v, f) for the entries (i, j), v f, of A B^T (A: M x K, B: NC x K,
// row-major with strides lda, ldb) that this lane computes; the 16 x 8 tiles
// are shared by the team's warps. SYRK: B = A, and only tiles that hold
// entries j <= i; the tiles on the diagonal use A's digits for both sides.
template <int TEAM, int K, bool SYRK, typename Out>
__device__ __forceinline__ void product(const Team<TEAM> &tm, const double *A, int lda, int M, const double *B,
                                        int ldb, int NC, Out out) {
  static_assert(TEAM >= 32, "whole warps");
  constexpr int KG = K / 8, W = TEAM / 32;
  const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int warp = tm.lane >> 5;
  const int MT = (M + 15) / 16, NT = (NC + 7) / 8;
  unsigned ad[2][KG][ND];
  int Ea[2] = {1, 1};
  int cur = -1;
#pragma unroll 1
  for (int item = warp; item < MT * NT; item += W) {
    const int mt = item / NT, nt = item - mt * NT;
    if (SYRK && nt * 8 > mt * 16 + 15) continue;
    if (mt != cur) {
      cur = mt;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (mt * 16 + h * 8 < M) {
          double x[KG][2];
          load_rows<K>(x, A, lda, mt * 16 + h * 8 + gid, M);
          Ea[h] = row_exponent<KG>(x);
#pragma unroll
          for (int g = 0; g < KG; ++g) digits(x[g][0], x[g][1], Ea[h], ad[h][g]);
        } else {
          Ea[h] = 1;
#pragma unroll
          for (int g = 0; g < KG; ++g)
#pragma unroll
            for (int i = 0; i < ND; ++i) ad[h][g][i] = 0u;
        }
      }
    }
    float c[ND][4];
    clear(c);
    int Eb;
    const int dg = SYRK ? nt - 2 * mt : -1;   // 0 or 1: the tile's columns are its own rows of half dg
    if (SYRK && dg >= 0) {
      Eb = dg ? Ea[1] : Ea[0];
#pragma unroll
      for (int g = 0; g < KG; ++g) {
        unsigned b[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) b[i] = dg ? ad[1][g][i] : ad[0][g][i];
        accumulate8(c, ad[0][g], ad[1][g], b);
      }
    } else {
      double x[KG][2];
      load_rows<K>(x, B, ldb, nt * 8 + gid, NC);
      Eb = row_exponent<KG>(x);
#pragma unroll
      for (int g = 0; g + 1 < KG; g += 2) {
        unsigned b[2][ND];
        digits(x[g][0], x[g][1], Eb, b[0]);
        digits(x[g + 1][0], x[g + 1][1], Eb, b[1]);
#pragma unroll
        for (int j = 0; j < ND; ++j)
#pragma unroll
          for (int i = 0; i + j < ND; ++i)
            mma_k16(c[i + j], ad[0][g][i], ad[1][g][i], ad[0][g + 1][i], ad[1][g + 1][i], b[0][j], b[1][j]);
      }
      if (KG % 2) {
        unsigned b[ND];
        digits(x[KG - 1][0], x[KG - 1][1], Eb, b);
        accumulate8(c, ad[0][KG - 1], ad[1][KG - 1], b);
      }
    }
    const int Eb0 = __shfl_sync(0xffffffffu, Eb, 8 * tig), Eb1 = __shfl_sync(0xffffffffu, Eb, 8 * tig + 4);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int i = mt * 16 + (t >> 1) * 8 + gid, j = nt * 8 + 2 * tig + (t & 1);
      const int up = up_scale(Ea[t >> 1]);
      const double val = assemble<K>(c, t, Ea[t >> 1] + up, (t & 1) ? Eb1 : Eb0);
      if (i < M && j < NC && (!SYRK || j <= i)) out(i, j, val, down_scale(up));
    }
  }
}

// lower(sD) -= X X^T (+ Y Y^T when Y != null).
template <int TEAM, int NB>
__device__ __forceinline__ void team_syrk_sub(const Team<TEAM> &tm, double *sD, const double *X, const double *Y) {
#pragma unroll 1
  for (int w = 0; w < (Y ? 2 : 1); ++w) {
    const double *P = w ? Y : X;
    // every entry is updated by the same lane in both passes
    product<TEAM, NB, true>(tm, P, NB, NB, P, NB, NB,
                            [&](int i, int j, double v, double f) { sD[i * NB + j] = fma(-v, f, sD[i * NB + j]); });
  }
}

// out (NB x NB, global) := -A B^T.
template <int TEAM, int NB>
__device__ __forceinline__ void team_gemm_nt_neg(const Team<TEAM> &tm, double *__restrict__ out, const double *A,
                                                 const double *B) {
  product<TEAM, NB, false>(tm, A, NB, NB, B, NB, NB,
                           [&](int i, int j, double v, double f) { out[i * NB + j] = -v * f; });
}

// 1 / d for a positive normal d to about an ulp: an FP32 estimate y of the
// reciprocal of the significand m (relative error e = 1 - m y below 2^-21),
// and the geometric series 1/m = y / (1 - e) cut after e^2, whose rest e^3 is
// below 2^-63, in FP64 (three dependent FP64 instructions; a library division
// takes more than twice that), the exponent by integer arithmetic.
// For d between 2^-1022 and 2^1022; d = 2^-1030 would give inf.
__device__ __forceinline__ double pivot_rcp(double d) {
  const int hi = __double2hiint(d);
  const int e = hi >> 20;
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(d));   // in [1, 2)
  // the significand's top 23 bits as a float
  const float mf = __uint_as_float(0x3f800000u | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)__double2loint(d) >> 29));
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(mf));   // in (0.5, 1]
  const unsigned yb = __float_as_uint(yf);
  const double y = __hiloint2double((int)((yb >> 3) + ((1023u - 127u) << 20)), (int)(yb << 29));
  const double err = fma(-m, y, 1.0);
  const double p = fma(err, err, err);
  const double r = fma(y, p, y);
  return __hiloint2double(__double2hiint(r) - ((e - 1023) << 20), __double2loint(r));
}

// Lower-triangle element e -> i | j << 8 for e < NB (NB + 1) / 2, one table per
// CTA (the arithmetic form, tri_index, costs a dozen instructions with a
// square root and two conversions for every element update).
template <int NB>
struct TriTable {
  unsigned short at[NB * (NB + 1) / 2];
};
template <int NB>
__device__ __forceinline__ void tri_fill(TriTable<NB> &t) {
  for (int e = threadIdx.x; e < NB * (NB + 1) / 2; e += blockDim.x) {
    int i, j;
    tri_index(e, i, j);
    t.at[e] = (unsigned short)(i | j << 8);
  }
}

// Cholesky of the block in sA (lower triangle read) by way of M D M^T: the
// pivots' reciprocals (three FP64 instructions on the critical path) drive
// the elimination (those near the ends of the range are scaled first, so that
// the reciprocal is a normal number), and the square roots of all pivots are
// taken at the end, one lane per column. On return the lower triangle holds L, the strict
// upper triangle the transpose of the unit factor M = L diag(L)^-1 (what
// the tail solves substitute with), and sInv[j] = 1/L_jj. A pivot that is
// not positive and finite is replaced by 1; returns 1 + its column, 0 if
// none.
template <int TEAM, int NB>
__device__ __forceinline__ int team_chol(const Team<TEAM> &tm, double *sA, double *sInv, const TriTable<NB> &tri) {
  int fail = 0;
#pragma unroll 1
  for (int j = 0; j < NB - 1; ++j) {
    double d = sA[j * NB + j];
    const int m = NB - 1 - j, ne = m * (m + 1) / 2;
    // unit(a) = a / d
    auto eliminate = [&](auto unit) {
      for (int i = j + 1 + tm.lane; i < NB; i += TEAM) sA[j * NB + i] = unit(sA[i * NB + j]);
      if (TEAM == 32) {
        tm.sync();
        for (int e = tm.lane; e < ne; e += TEAM) {
          const int ab = tri.at[e], i = j + 1 + (ab & 255), k = j + 1 + (ab >> 8);
          sA[i * NB + k] = fma(-sA[j * NB + i], sA[k * NB + j], sA[i * NB + k]);
        }
      } else {
        // several warps: each element scales its own row entry again (the
        // same product) instead of waiting for the column at a barrier
        for (int e = tm.lane; e < ne; e += TEAM) {
          const int ab = tri.at[e], i = j + 1 + (ab & 255), k = j + 1 + (ab >> 8);
          sA[i * NB + k] = fma(-unit(sA[i * NB + j]), sA[k * NB + j], sA[i * NB + k]);
        }
      }
    };
    // (the same for the whole team)
    if ((unsigned)(__double2hiint(d) - (64 << 20)) < (1900u << 20)) {
      const double r = pivot_rcp(d);
      eliminate([&](double a) { return a * r; });
    } else {   // not positive and finite, or 1/d could overflow or be subnormal
      if (!pivot_ok(d)) {
        if (!fail) fail = j + 1;
        d = 1.0;
      }
      const double t = d < 1.0 ? 0x1p64 : 0x1p-64, r = pivot_rcp(d * t);
      eliminate([&](double a) { return (a * t) * r; });
    }
    tm.sync();
  }
  if (!pivot_ok(sA[NB * NB - 1]) && !fail) fail = NB;
  for (int j = tm.lane; j < NB; j += TEAM) {
    double d = sA[j * NB + j];
    if (!pivot_ok(d)) d = 1.0;
    sInv[j] = rsqrt(d);
  }
  tm.sync();
  constexpr int NE = NB * (NB + 1) / 2;
  for (int e = tm.lane; e < NE; e += TEAM) {
    const int ij = tri.at[e], i = ij & 255, j = ij >> 8;
    double v = sA[i * NB + j];
    if (i == j && !pivot_ok(v)) v = 1.0;
    sA[i * NB + j] = v * sInv[j];
  }
  tm.sync();
  return fail;
}

// Column l of a panel in a scale-free form. The variables of a stage may have
// different units: with K = S K' S (S diagonal) column l of a coupling block
// carries s_l and column l of L_pp^-1 carries 1/s_l, while a digit product is
// exact relative to the largest entries of its two rows only. Both rows are
// brought to one scale each by the power of two 2^o_l next to L_ll, from the
// exponent of 1/L_ll: y_l 2^-o_l (an offset of the exponents below) and
// (L_pp^-1)_kl 2^o_l, both exact. Without it the backward error of the solve
// grew with the spread of the units within a panel (emulated, 1e-16 at 2^0,
// 1e-12 at 2^20, 2e-9 at 2^30). With the offsets
// read before the tiles it costs nothing at S = 512, N = 128, nb = 24 (factor and solve
// 3727 us without it, 3684 with; read in every tile 3782).
__device__ __forceinline__ int column_scale(double inv) { return 1023 - (__double2hiint(inv) >> 20); }   // (inv > 0)

// Largest biased exponents E0, E1 of a panel's rows y0 (rows 0-7) and y1 (8-15), whose
// entries in the lane's two columns count as x 2^-o0 and x 2^-o1; kBadRow as
// in row_exponent.
__device__ __forceinline__ void row_exponents_scaled(const double (&y0)[2], const double (&y1)[2], int o0, int o1,
                                                     int &E0, int &E1) {
  const double x[4] = {y0[0], y0[1], y1[0], y1[1]};
  int c[4];
  unsigned mx = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const unsigned u = ((unsigned)__double2hiint(x[t]) & 0x7fffffffu) - 0x100000u;   // zero and subnormal wrap around
    mx = max(mx, u);
    c[t] = (int)(u >> 20) + 1 - (t & 1 ? o1 : o0);
  }
  if (mx >= 0x7fe00000u) {   // an entry that is not a normal number
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int h = __double2hiint(x[t]) & 0x7fffffff;
      if (h >= 0x7ff00000) c[t] = kBadRow;
      if (h < 0x100000) c[t] = (h | __double2loint(x[t])) ? 1 - (t & 1 ? o1 : o0) : -4096;
    }
  }
  E0 = max(c[0], c[1]);
  E1 = max(c[2], c[3]);
#pragma unroll
  for (int m = 1; m <= 2; m <<= 1) {
    E0 = max(E0, __shfl_xor_sync(0xffffffffu, E0, m));
    E1 = max(E1, __shfl_xor_sync(0xffffffffu, E1, m));
  }
}

// G_p = (L_pp)^-1 diag(p_l) for the 8 x 8 diagonal blocks of L, in place of
// those blocks (zeros above the diagonal): L_pp^-1 = diag(1/L_jj) M_pp^-1 with
// the unit factor M. One lane per column substitutes with M_pp (28 FMAs, all
// panels at once), from p_l instead of 1 (column_scale).
template <int TEAM, int NB>
__device__ __forceinline__ void team_invert_diagonal(const Team<TEAM> &tm, double *sA, const double *inv) {
#pragma unroll
  for (int cb = 0; cb < NB; cb += TEAM) {
    const int c = cb + tm.lane, c0 = c & ~7, jj = c & 7;
    double v[8];
    if (c < NB) {
      const double *M = sA + c0 * NB + c0;   // M_kl at M[l * NB + k], l < k
      const double p = __hiloint2double((1023 + column_scale(inv[c])) << 20, 0);
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = k == jj ? p : 0.0;
#pragma unroll
      for (int k = 1; k < 8; ++k) {
        double acc = 0.0;
#pragma unroll
        for (int l = 0; l < k; ++l) acc = fma(-M[l * NB + k], v[l], acc);
        if (k > jj) v[k] = acc;
      }
    }
    tm.sync();
    if (c < NB) {
#pragma unroll
      for (int k = 0; k < 8; ++k) sA[(c0 + k) * NB + c] = v[k] * inv[c0 + k];
    }
    tm.sync();
  }
}

// One panel of team_trsm_lt for 16 rows held in registers (x[h][g]: rows 0-7
// and 8-15 of the tile): the columns before the panel act on it through the
// lower triangle of L, then it is multiplied by the inverse of its diagonal
// block, both scaled per column (column_scale; o: this lane's offsets). The accumulators of a product
// have the layout of the next one's operand, so nothing passes through shared
// memory in between.
template <int NB, int P>
__device__ __forceinline__ void trsm_panel(double (&x)[2][NB / 8][2], const double *sA, const int (&o)[NB / 8]) {
  constexpr int c0 = 8 * P;
  const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  if constexpr (P > 0) {
    const int E0 = row_exponent<P>(x[0]), E1 = row_exponent<P>(x[1]);
    double b[P][2];
    load_rows<c0>(b, sA + c0 * NB, NB, gid, 8);
    const int Eb = row_exponent<P>(b);
    float c[ND][4];
    clear(c);
#pragma unroll
    for (int g = 0; g + 1 < P; g += 2) {
      unsigned a0[2][ND], a1[2][ND], bd[2][ND];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        digits(x[0][g + u][0], x[0][g + u][1], E0, a0[u]);
        digits(x[1][g + u][0], x[1][g + u][1], E1, a1[u]);
        digits(b[g + u][0], b[g + u][1], Eb, bd[u]);
      }
      accumulate16(c, a0, a1, bd);
    }
    if (P % 2) {
      unsigned a0[ND], a1[ND], bd[ND];
      digits(x[0][P - 1][0], x[0][P - 1][1], E0, a0);
      digits(x[1][P - 1][0], x[1][P - 1][1], E1, a1);
      digits(b[P - 1][0], b[P - 1][1], Eb, bd);
      accumulate8(c, a0, a1, bd);
    }
    const int Eb0 = __shfl_sync(0xffffffffu, Eb, 8 * tig), Eb1 = __shfl_sync(0xffffffffu, Eb, 8 * tig + 4);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int E = t >> 1 ? E1 : E0, up = up_scale(E);
      x[t >> 1][P][t & 1] = fma(-assemble<c0>(c, t, E + up, (t & 1) ? Eb1 : Eb0), down_scale(up), x[t >> 1][P][t & 1]);
    }
  }
  double b[1][2];
  load_rows<8>(b, sA + c0 * NB + c0, NB, gid, 8);
  const int Eb = row_exponent<1>(b);
  const int o0 = o[P] >> 16, o1 = (int)(short)o[P];
  int E0, E1;
  row_exponents_scaled(x[0][P], x[1][P], o0, o1, E0, E1);
  unsigned a0[ND], a1[ND], bd[ND];
  digits(x[0][P][0], x[0][P][1], E0 + o0, E0 + o1, a0);
  digits(x[1][P][0], x[1][P][1], E1 + o0, E1 + o1, a1);
  digits(b[0][0], b[0][1], Eb, bd);
  float c[ND][4];
  clear(c);
  accumulate8(c, a0, a1, bd);
  const int Eb0 = __shfl_sync(0xffffffffu, Eb, 8 * tig), Eb1 = __shfl_sync(0xffffffffu, Eb, 8 * tig + 4);
#pragma unroll
  for (int t = 0; t < 4; ++t)   // (entries of X: against sqrt(K_ii) > 2^-538 a subnormal one does not show)
    x[t >> 1][P][t & 1] = assemble<8>(c, t, t >> 1 ? E1 : E0, (t & 1) ? Eb1 : Eb0);
  if constexpr (c0 + 8 < NB) trsm_panel<NB, P + 1>(x, sA, o);
}

// X (M x NB) := X L^{-T}, all of it sliced products, 16 rows per warp at a
// time. sA as team_chol leaves it; its diagonal 8 x 8 blocks are overwritten
// (the factor is stored before).
template <int TEAM, int NB>
__device__ __forceinline__ void team_trsm_lt(const Team<TEAM> &tm, double *X, int M, double *sA, const double *inv) {
  constexpr int KG = NB / 8;
  const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  tm.sync();
  team_invert_diagonal<TEAM, NB>(tm, sA, inv);
  int o[KG];   // the column offsets of this lane in every panel, two to a word
#pragma unroll
  for (int g = 0; g < KG; ++g)
    o[g] = column_scale(inv[8 * g + 2 * tig]) << 16 | (column_scale(inv[8 * g + 2 * tig + 1]) & 0xffff);
#pragma unroll 1
  for (int mt = tm.lane >> 5; mt * 16 < M; mt += TEAM / 32) {
    double x[2][KG][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) load_rows<NB>(x[h], X, NB, mt * 16 + h * 8 + gid, M);
    trsm_panel<NB, 0>(x, sA, o);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = mt * 16 + h * 8 + gid;
#pragma unroll
      for (int g = 0; g < KG; ++g) {
        const int k = 8 * g + 2 * tig;
        if (row < M)
          *reinterpret_cast<double2 *>(X + row * NB + k) = make_double2(x[h][g][0], x[h][g][1]);
      }
    }
  }
  tm.sync();
}

}  // namespace sliced
}  // namespace bm
