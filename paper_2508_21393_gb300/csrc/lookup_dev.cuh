// Device helpers of the lookup-argument kernels (kernels_lookup.cu: start,
// tables, transcript steps, tails; kernels_lookup_pass.cu: the batched round
// passes), shared by both translation units.
//
// The four sums a round needs, per pair (k, k + h) with f = eq(u_{t+1..L}, k):
//   T(X) = sum f (A S')(X)   A(X) = sum A(X)   U(X) = sum f (B T')(X)   V(X) = sum (B m)(X)
// (U, V in the table rounds only).  A is linear, the others quadratic in X, and
// each has a running claim, its value at the last challenge: A(0) + A(1) and
// V(0) + V(1) are theirs, and (1 - u_t) T(0) + u_t T(1), (1 - u_t) U(0) + u_t U(1)
// those of T, U (the same split of the eq factor as in A. Gruen, "Some
// Improvements for the PIOP for ZeroCheck", IACR ePrint 2024/108).  So a pass
// sums only the values at 0 and the leading coefficients (index "inf"): for T
// two products per pair instead of three.  What else a pair does not need:
//  * T(0) = T(1) = 1 in round 1 and U(0) = U(1) = 1 in the first table round
//    (A S' = B T' = 1 on unfolded entries and the eq factors sum to 1);
//  * S' differs between table entries by a small integer, and A S' = 1: round
//    1's leading term is f (a1 - a0)(j1 - j0); round 2 needs S' only in the
//    difference of a pair, and its T(0) is 1 - r (1 - r) sum f (a' - a)(j' - j)
//    over the entries a, a' that fold into a pair's first; round 3 forms S'
//    from the four table indices and the four eq weights of (r_1, r_2): products
//    by integers of 16 to 18 bits throughout;
//  * round 2's folded A comes from the tables (1 - r) B, r B (two products per
//    table entry instead of two per pair);
//  * T'(k) = beta + t0 + k is affine in k: folded it is Tb[k] + toff, and its
//    leading coefficient the constant h;
//  * sums of products are reduced once per thread (wide_mac).
#pragma once
#include "prologue_dev.cuh"
#include "rounds_dev.cuh"

namespace vl {

namespace {

constexpr uint8_t LBL_BETA = 'b', LBL_ALPHA = 'a';
constexpr int LK_STEP_THREADS = 128;  // transcript step: its message schedules take warps 1 to 3
constexpr int LK_MAX_WARPS = 16;
constexpr int LK_CL_PAIRS = 8 * RND_MAX_CTAS;  // pairs of a round spread over a cluster, at least

// Table index of cube entry k, as the histogram pass left it: S's layout, the
// offset t0 and the padding are dealt with once per entry there, not at each of its
// uses in rounds 1 to 3 (passes of the 512 lookups of a 7B step 402, 892, 675 ->
// 340, 725, 554 us, the histogram pass 43 -> 57).
__device__ __forceinline__ int lk_table_index(const LkDev& L, int k) { return L.idx[k]; }

__device__ __forceinline__ Fr lk_fold(const Fr& x0, const Fr& x1, const Fr& r) {
  return fr_add(x0, mont_mul_ni(r, fr_sub(x1, x0)));
}

// a d mod r for a signed integer |d| < 2^18.
__device__ __forceinline__ Fr lk_times(const Fr& a, int d) {
  const Fr z = small_mul_mod(a, (uint32_t)(d < 0 ? -d : d));
  return d < 0 ? fr_neg(z) : z;
}

// S' at entry k of the cube folded by r_1 and r_2 (2^q entries): beta + t0 +
// sum_b w4[b] j(k + b 2^q).
__device__ __forceinline__ Fr lk_s_round3(const LkDev* L, int k, int q) {
  uint32_t t[9], z[9];
  small_mul(t, L->w4[0].v, (uint32_t)lk_table_index(*L, k));
#pragma unroll
  for (int b = 1; b < 4; b++) {
    small_mul(z, L->w4[b].v, (uint32_t)lk_table_index(*L, k + (b << q)));
    add9(t, z);
  }
  return fr_add(L->Tb[0], small_reduce(t));
}

// Sums of one thread's pairs, A side: T(0), T(inf), A(0).
struct LkSumA {
  uint32_t t0[17], ti[17], a0[9];
  __device__ __forceinline__ void zero() {
    wide_zero(t0), wide_zero(ti);
#pragma unroll
    for (int i = 0; i < 9; i++) a0[i] = 0;
  }
  __device__ __forceinline__ void columns(unsigned long long (&col)[3][8]) const {
    wide_redc(t0, col[0]);
    wide_redc(ti, col[1]);
    sum9_columns(a0, col[2]);
  }
};
// Table side: U(0), U(inf) / h, V(0), V(inf).
struct LkSumB {
  uint32_t u0[17], ui[17], v0[17], vi[17];
  __device__ __forceinline__ void zero() { wide_zero(u0), wide_zero(ui), wide_zero(v0), wide_zero(vi); }
  __device__ __forceinline__ void columns(unsigned long long (&col)[4][8]) const {
    wide_redc(u0, col[0]);
    wide_redc(ui, col[1]);
    wide_redc(v0, col[2]);
    wide_redc(vi, col[3]);
  }
};

// One pair (k, k + h) of round t, r = r_(t-1), A side.  MODE 0: round 1, from the unfolded
// cube; 1: round 2, A folded on the fly and written, t0 summing Q = f (a' - a)(j'
// - j) (T(0) = 1 - r (1 - r) Q); 2: round 3, A folded in place, S' formed and
// written; 3: later rounds, both folded in place.
template <int MODE>
__device__ __forceinline__ void lk_pair_a(LkDev* L, int k, int h, const Fr& f, const Fr& r, LkSumA& s) {
  if constexpr (MODE == 0) {
    const int j0 = lk_table_index(*L, k), j1 = lk_table_index(*L, k + h), d = j1 - j0;
    const Fr a0 = L->Binv[j0], a1 = L->Binv[j1];
    sum9_add(s.a0, a0);
    // (a1 - a0)(s1 - s0) = (a1 - a0)(j1 - j0), both signs flipped for j1 < j0
    wide_mac_small(s.ti, f, d < 0 ? fr_sub(a0, a1) : fr_sub(a1, a0), (uint32_t)(d < 0 ? -d : d));
  } else if constexpr (MODE == 1) {
    const int j0 = lk_table_index(*L, k), j1 = lk_table_index(*L, k + h);
    const int j2 = lk_table_index(*L, k + 2 * h), j3 = lk_table_index(*L, k + 3 * h);
    const Fr b0 = L->Binv[j0], b2 = L->Binv[j2];
    Fr a0, a1;
    if (L->round2) {
      a0 = fr_add(L->UB[j0], L->VB[j2]);
      a1 = fr_add(L->UB[j1], L->VB[j3]);
    } else {
      a0 = lk_fold(b0, b2, r);
      a1 = lk_fold(L->Binv[j1], L->Binv[j3], r);
    }
    L->VA[k] = a0, L->VA[k + h] = a1;
    sum9_add(s.a0, a0);
    const int d = j2 - j0;
    wide_mac_small(s.t0, f, d < 0 ? fr_sub(b0, b2) : fr_sub(b2, b0), (uint32_t)(d < 0 ? -d : d));
    // s1 - s0 = (j1 - j0) + r ((j3 - j2) - (j1 - j0))
    const Fr ds = fr_add(lk_times(fr_r1(), j1 - j0), lk_times(r, (j3 - j2) - (j1 - j0)));
    wide_mac(s.ti, f, mont_mul_ni(fr_sub(a1, a0), ds));
  } else {
    const Fr a0 = lk_fold(L->VA[k], L->VA[k + 2 * h], r);
    const Fr a1 = lk_fold(L->VA[k + h], L->VA[k + 3 * h], r);
    Fr s0, s1;
    if constexpr (MODE == 2) {
      s0 = lk_s_round3(L, k, L->L - 2);
      s1 = lk_s_round3(L, k + h, L->L - 2);
    } else {
      s0 = lk_fold(L->VS[k], L->VS[k + 2 * h], r);
      s1 = lk_fold(L->VS[k + h], L->VS[k + 3 * h], r);
    }
    L->VA[k] = a0, L->VA[k + h] = a1;
    L->VS[k] = s0, L->VS[k + h] = s1;
    sum9_add(s.a0, a0);
    wide_mac(s.t0, f, mont_mul_ni(a0, s0));
    wide_mac(s.ti, f, mont_mul_ni(fr_sub(a1, a0), fr_sub(s1, s0)));
  }
}

// One pair of a table round (round tj of the last log2 N; eq(u_low, .) folded
// by the bound table variables is the A side's factor f times a scalar of the
// transcript step): B and m are folded in place after the first table round.
__device__ __forceinline__ void lk_pair_b(LkDev* L, int tj, int k, int h, const Fr& f, const Fr& r, const Fr& toff,
                                          LkSumB& s) {
  Fr b0, b1, m0, m1;
  if (tj == 1) {
    b0 = L->WB[k], b1 = L->WB[k + h];
    m0 = L->WM[k], m1 = L->WM[k + h];
  } else {
    b0 = lk_fold(L->WB[k], L->WB[k + 2 * h], r);
    b1 = lk_fold(L->WB[k + h], L->WB[k + 3 * h], r);
    m0 = lk_fold(L->WM[k], L->WM[k + 2 * h], r);
    m1 = lk_fold(L->WM[k + h], L->WM[k + 3 * h], r);
    L->WB[k] = b0, L->WB[k + h] = b1;
    L->WM[k] = m0, L->WM[k + h] = m1;
    wide_mac(s.u0, f, mont_mul_ni(b0, fr_add(L->Tb[k], toff)));
  }
  const Fr db = fr_sub(b1, b0);
  wide_mac(s.ui, f, db);
  wide_mac(s.v0, b0, m0);
  wide_mac(s.vi, db, fr_sub(m1, m0));
}

// Where round t reads eq(u_{t+1..L}, k): hiP[k >> sE] . loP_sE[k mod 2^sE]
// while t binds one of the first L - sE variables (high), loP_(L-t)[k] after.
struct LkEq {
  const Fr* f_tab;
  const Fr* hi_tab;
  int f_mask;
  bool high;
  __device__ LkEq(const LkDev* L, int t) {
    high = t <= L->L - L->sE;
    const int mask = (1 << L->sE) - 1;
    f_tab = high ? L->loP + mask : L->loP + (1 << (L->L - t)) - 1;
    f_mask = high ? mask : (1 << (L->L - t)) - 1;
    hi_tab = L->hiP + (high ? (1 << (L->L - L->sE - t)) - 1 : 0);
  }
};

}  // namespace

}  // namespace vl
