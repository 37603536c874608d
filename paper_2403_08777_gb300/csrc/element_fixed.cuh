// The element routines of element.cuh in block fixed-point arithmetic
// (fixed.cuh): the same restructured form, its products on the integer pipe.
//
// Scaling. Every index carries its own power of two, so that flat cells and
// velocity components of different size keep their relative accuracy:
//   D_k,i  = u_k,i - u_0,i   2^ed_i      (exact differences, normalised per i)
//   C_k,j  (k = 1..3)        2^t_j       (cofactor vectors, per axis j)
//   G_i,j                    2^(eG_i + t_j)
//   W_g,j  = u_g,j + beta S_j; the Gauss point velocity is alpha W_g, with
//            alpha = 1/sqrt 5 and beta = (sqrt 5 - 1)/4. Wherever it is
//            contracted with an axis index, W~_g,j in units 2^(kap - t_j),
//            kap = max_j (eu_j + t_j), so that sum_j C_a,j W~_g,j needs no
//            alignment; its norm |W_g|^2 uses one exponent for all j.
// Contractions over an axis then cancel t_j, and only sums of different terms
// (convection, viscosity, pressure, stabilisation) are aligned, row by row.
// The 4 square roots and 4 reciprocals of tau stay on the FP64 pipe, which
// works beside the integer pipe.
//
// Code size. Written out, the routine is about 4600 instructions; GB300's
// instruction supply falls from 0.93 to 0.3 - 0.65 instructions per clock and
// sub-partition once a loop body exceeds about 32 KB (2048 instructions). The
// loops over components, Gauss points and rows are therefore kept rolled,
// their per-thread arrays in shared memory.
//
// Elements whose data are outside 2^-100 .. 2^100 (or not finite), and those
// with a gradient that vanishes on the axis that decides an alignment
// (aligned_rows), are left to the FP64 routines: the functions return false
// before writing anything.
#pragma once

#include "element.cuh"
#include "fixed.cuh"

namespace nsrhs {
namespace fixed {

// A launch-uniform scalar: m 2^(e - B), |m| < 2^B, B = 60 where it is the
// first operand of mul8, 61 elsewhere.
struct Scalar {
  Limb m;
  int e;
};

// Launch-uniform parameters (host: make_fixed_params).
struct FixedParams {
  ElemParams<double> P;  // for the FP64 routines
  double c1mu;           // c1 mu
  double k2;             // c2 rho
  double k2a;            // c2 rho alpha
  double rhoc;           // rho c_vreman
  Scalar a2;             // -rho^2 alpha^2 / 24
  Scalar a1;             // -mu / 6
  Scalar b4;             // -rho alpha / 24
  Scalar m120;           // -rho / 120 (skew: -rho / 240), B = 60
  Scalar r48;            // rho alpha^2 / 48, B = 60
  bool in_range;         // every parameter 0 or within 2^-60 .. 2^60
};

constexpr int64_t kBeta62 = 0x13c6ef372fe94f83ll;       // beta 2^62
constexpr int64_t kBeta61 = 0x9e3779b97f4a7c2ll;        // beta 2^61
constexpr int64_t kQB61 = 0x46c1b47480244d9ll;          // QB 2^61
constexpr int64_t kEightFifteenths60 = 0x888888888888889ll;  // (8/15) 2^60
constexpr int64_t kTwoThirds61 = 0x1555555555555555ll;  // (2/3) 2^61; 1/24 = 2^-4 2/3

// Per-thread scratch in shared memory: 64-bit slots and 16-bit words (for
// exponents), the same slot of the block's THREADS threads side by side (no
// bank conflicts). Rolled loops index it at run time.
constexpr int kFwdSlots = 49;   // 64-bit slots of element_rhs_fixed
constexpr int kFwdSlotsSkew = 61;
constexpr int kFwdWords = 15;   // 16-bit words

template <int THREADS>
struct Scratch {
  int64_t* q;  // + threadIdx.x
  int16_t* w;
  __device__ __forceinline__ int64_t get(int s) const { return q[s * THREADS]; }
  __device__ __forceinline__ void put(int s, int64_t x) const { q[s * THREADS] = x; }
  __device__ __forceinline__ Limb limb(int s) const {
    const uint64_t x = (uint64_t)q[s * THREADS];
    return {(int32_t)(x >> 32), (int32_t)x};
  }
  __device__ __forceinline__ void put(int s, const Limb& a) const {
    q[s * THREADS] = (int64_t)((uint64_t)(uint32_t)a.h << 32 | (uint32_t)a.l);
  }
  __device__ __forceinline__ double real(int s) const { return make_double((uint64_t)q[s * THREADS]); }
  __device__ __forceinline__ void put_real(int s, double x) const {
    q[s * THREADS] = (int64_t)((uint64_t)(uint32_t)hi_word(x) << 32 | lo_word(x));
  }
  __device__ __forceinline__ int32_t word(int s) const { return w[s * THREADS]; }
  __device__ __forceinline__ void put_word(int s, int32_t x) const { w[s * THREADS] = (int16_t)x; }
};

// Slots. C: cofactors (input c_k,j, k = 1..3, at kSlotC + 3 (k - 1) + j, then
// the limbs of C_k,j). U: nodal values (input component i of node a at
// kSlotU + 4 i + a, i = 3 the pressure; then W, then W~). X: tau W~ (from the
// pressure's input slots on). G: gradient rows, row 3 the pressure's. S: sums
// over the nodes.
enum : int { kSlotC = 0, kSlotU = 9, kSlotX = 21, kSlotG = 33, kSlotS = 45, kSlotW = 49 };
enum : int { kWordT = 0, kWordEu = 3, kWordEg = 7, kWordX = 11 };

// beta S for S a sum of nodal values, |S| < 2^61.
__device__ __forceinline__ int64_t beta_sum(int64_t S) {
  constexpr Limb b = limb(kBeta62);  // 4 S (beta 2^62) / 2^64
  const Limb s = limb(S);
  int64_t M = mad_wide(s.h, b.l, 1ll << 31);
  M = mad_wide(s.l, b.h, M);
  return mad_wide(hi32(M), 4, mad_wide(s.h, b.h * 4, 0));
}

// beta V, |V| < 2^62.4 (a sum of four W~), below 2^60.7.
__device__ __forceinline__ int64_t beta_sum_wide(int64_t V) {
  return mulx<3>(limb(kBeta61), limb(V >> 2)) * 4;
}

// QB V, likewise.
__device__ __forceinline__ int64_t qb_sum(int64_t V) {
  return mulx<3>(limb(kQB61), limb(V >> 2)) * 4;
}

// |v|^2 of the vector v_i 2^(eu_i - 59), |v_i| < 2^60.2, as a double;
// eum = max eu_i. The vector is normalised first: a Gauss point may be nearly
// at rest.
__device__ __forceinline__ double velocity_norm2(int64_t v0, int64_t v1, int64_t v2,
                                                 const int eu[3], int eum) {
  const int64_t x0 = shr(v0, eum - eu[0]), x1 = shr(v1, eum - eu[1]), x2 = shr(v2, eum - eu[2]);
  const int n = norm_shift(mag(x0) | mag(x1) | mag(x2));
  return to_double(square3(limb(shl(x0, n)), limb(shl(x1, n)), limb(shl(x2, n))),
                   2 * (eum - n + 3));
}

// Sums over an axis, of a gradient row R with itself scaled (viscosity, terms 2 t_j)
// or with the velocity (convection, terms eu_j + t_j, twice in tau's part), are
// aligned to the largest term that there may be. Against a 53-bit number that costs
// nothing, since the double-precision sum has a rounding error of that size, unless
// the row is 0 on that axis, as where a field does not vary across flat cells or
// along the stream: then the double-precision sum may be as exact as its other
// terms. Whether no row loses more bits in this way than a 59-bit number has to spare
// (cells flatter than 8 with such a field do); rows at slot sR, n of them, those
// from v on (three) also taken with the velocity. least: the smallest mag() of an
// entry; rows without a 0, the usual case, need no look.
constexpr int kSpare = 6;
template <int THREADS>
__device__ __forceinline__ bool aligned_rows(const Scratch<THREADS>& sc, int sR, int n, int v,
                                             const int eu[3], const int t[3], int tmax,
                                             uint32_t least) {
  // the warp takes the branch together: threads that took it alone would do the
  // rest of the element alone (16^3 step 55 -> 69 us)
  if (!any_lane(least == 0u)) return true;
  int w[3], hi = -30000, lost = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    w[j] = eu[j] > kRestExp ? eu[j] + t[j] : -30000;
    hi = imax(hi, w[j]);
  }
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    int at = -30000, aw = -30000;
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (mag(sc.get(sR + 3 * i + j)) > 1u) at = imax(at, t[j]), aw = imax(aw, w[j]);
    if (at > -30000) lost = imax(lost, 2 * (tmax - at));
    if (aw > -30000 && (unsigned)(i - v) < 3u) lost = imax(lost, 2 * (hi - aw));
  }
  return lost <= kSpare;
}

// From the accumulated Q = sum tau W~ W~^T and T = sum tau W~ (T in units
// 2^(theta + kap - t_j - 58)): Qp = a2 Q + a1 I (real 2^(eP - 60 - t_k - t_j);
// 00 11 22 01 02 12) and sT = b4 T (real 2^(eT - 60 - t_j)).
__device__ __forceinline__ void gauss_matrices(const Acc q[6], int64_t T[3], int theta, int kap,
                                               const Limb& inv, int einv, int64_t a1, int ea1,
                                               const int t[3], int tmax, const FixedParams& P,
                                               Limb Qp[6], int& eP, Limb sT[3], int& eT) {
  int64_t qf[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) qf[k] = fin(q[k]);
  // real qf 2^(theta + 2 kap - t_k - t_j - 53), qf < 2^58.2; Q is positive
  // semidefinite: its diagonal bounds it
  const int nq = norm_shift(mag(qf[0]) | mag(qf[1]) | mag(qf[2]));
  const Limb a2 = limb(mul8(inv, P.a2.m));
  const int e2 = P.a2.e + einv + theta + 2 * kap + 8 - nq;
  eP = imax(e2, ea1 + 2 * tmax) + 1;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    int64_t x = shr(mul8(a2, limb(shl(qf[k], nq))), eP - e2);
    if (k < 3) x += shr(a1, eP - ea1 - 2 * t[k]);
    Qp[k] = limb(x);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) T[j] >>= 1;  // < 2^61
  const int nt = norm_shift(mag(T[0]) | mag(T[1]) | mag(T[2]));
  const Limb b4 = limb(mul8(inv, P.b4.m));
#pragma unroll
  for (int j = 0; j < 3; ++j) sT[j] = limb(mul8(b4, limb(shl(T[j], nt))));
  eT = P.b4.e + einv + theta + kap + 4 - nt;
}

// The row base + sum_j K_j C_a,j with base = +-tr R / 24 (third = +-(2/3) 2^60)
// and K_j = sum_k sT_k R_jk + sg r_j, from the rows R at slot sR (exponents
// eR_j + t_k) and the vector r at slot sr (exponents t_j and, with sg's, er).
// sE, sT0: the words of eR and t; sk: three free slots. Returns the exponent
// for to_double.
template <int THREADS>
__device__ __forceinline__ int trace_row(const Scratch<THREADS>& sc, int sR, int sr, int sE, int sT0,
                                         const int eR[3], const int t[3], int tmax,
                                         const Limb sT[3], int eT, const Limb& sg, int er,
                                         int64_t third, int sk, Limb K[3],
                                         int64_t& base) {
  // tr R, often much smaller than its terms: summed unshifted (below 2^62.6)
  // and normalised
  const int et = imax(eR[0] + t[0], imax(eR[1] + t[1], eR[2] + t[2]));
  int64_t tr = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) tr += shr(sc.get(sR + 4 * j), et - (eR[j] + t[j]));
  const int nt = norm_shift(mag(tr));
  tr = shl(tr, imax(nt, 0)) >> imax(-nt, 0);
  // tr R / 24 = (tr / 3) 2^(ec - 56)
  const int64_t c0 = mul8(limb(third), limb(tr));
  const int ec = et - nt - 8;
  int e = imax(ec, er + 2 * tmax);
#pragma unroll
  for (int j = 0; j < 3; ++j) e = imax(e, eR[j] + t[j] + eT);
  uint32_t m = 0;
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    Limb g[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) g[i] = limb(sc.get(sR + 3 * j + i));
    const int tj = sc.word(sT0 + j);
    const int64_t k =
        shr(dot3x<2>(sT[0], g[0], sT[1], g[1], sT[2], g[2]), e - (sc.word(sE + j) + eT + tj)) +
        shr(mulx<2>(sg, limb(sc.get(sr + j))), e - (er + 2 * tj));
    m |= mag(k);
    sc.put(sk + j, k);
  }
  base = shr_round(c0, e - ec);  // the K_j may cancel in sum_j K_j C_a,j
  // |k| < 2^61, |base| < 2^60
  const int n = norm_shift(m | mag(base));
  base = shl(base, n);
#pragma unroll
  for (int j = 0; j < 3; ++j) K[j] = limb(shl(sc.get(sk + j), n));
  return e - n + 4;
}

// Vreman's eddy viscosity from detJ grad u (element.cuh), on the FP64 pipe.
__device__ __forceinline__ void vreman_invariants(const double g[3][3], double b[6], double& A,
                                                  double& B) {
  b[0] = fmac(g[0][2], g[0][2], fmac(g[0][1], g[0][1], g[0][0] * g[0][0]));
  b[1] = fmac(g[1][2], g[1][2], fmac(g[1][1], g[1][1], g[1][0] * g[1][0]));
  b[2] = fmac(g[2][2], g[2][2], fmac(g[2][1], g[2][1], g[2][0] * g[2][0]));
  b[3] = fmac(g[0][2], g[1][2], fmac(g[0][1], g[1][1], g[0][0] * g[1][0]));
  b[4] = fmac(g[0][2], g[2][2], fmac(g[0][1], g[2][1], g[0][0] * g[2][0]));
  b[5] = fmac(g[1][2], g[2][2], fmac(g[1][1], g[2][1], g[1][0] * g[2][0]));
  A = (b[0] + b[1]) + b[2];
  B = fmac(b[1], b[2], -(b[5] * b[5]));
  B = fmac(b[0], b[2], fmac(-b[4], b[4], B));
  B = fmac(b[0], b[1], fmac(-b[3], b[3], B));
}
__device__ __forceinline__ void vreman_viscosity(const double g[3][3], double rh,
                                                 const FixedParams& P, double& A, double& phi,
                                                 double& scale, double& mu_eff, bool& active) {
  using M = MathOps<double>;
  double b[6], B;
  vreman_invariants(g, b, A, B);
  if (A > 0.0 && B > 0.0) {
    active = true;
    scale = P.rhoc * rh;
    phi = M::sqrt_(B * M::rcp(A));
    mu_eff = fmac(scale, phi, P.P.mu);
  }
}
// Its part of Gbar: mub scale / (phi A) (tr(beta) I - beta - phi^2 I) Gh.
template <class Get>
__device__ __forceinline__ void vreman_gradient(const Get& get, double mub, double A, double phi,
                                                double scale, double D[3][3]) {
  double g[3][3], b[6], A2, B2;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) g[i][j] = get(i, j);
  vreman_invariants(g, b, A2, B2);
  const double f = mub * scale * MathOps<double>::rcp(phi * A);
  const double t = f * (A - phi * phi);
  const double m01 = -f * b[3], m02 = -f * b[4], m12 = -f * b[5];
  const double m[3][3] = {{fmac(-f, b[0], t), m01, m02},
                          {m01, fmac(-f, b[1], t), m12},
                          {m02, m12, fmac(-f, b[2], t)}};
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      D[i][j] = fmac(m[i][2], g[2][j], fmac(m[i][1], g[1][j], m[i][0] * g[0][j]));
}

template <int FLAGS, int THREADS, class Out>
__device__ __forceinline__ bool element_rhs_fixed(const Scratch<THREADS>& sc, double inv_det,
                                                  double rh, const FixedParams& P,
                                                  const Out& out) {
  using M = MathOps<double>;
  constexpr bool VREMAN = (FLAGS & kVreman) != 0;
  constexpr bool SKEW = (FLAGS & kSkew) != 0;
  constexpr bool TAUE = (FLAGS & kTauElem) != 0;
  constexpr int kSlotWt = SKEW ? kSlotW : kSlotU;  // W~: in place of W where W is not needed again
  // ---- cofactor vectors: real C 2^(t_j - 61) ----
  bool ok = (uint32_t)((hi_word(inv_det) >> 20) - 723) <= 600u &&
            (uint32_t)((hi_word(rh) >> 20) - 823) <= 400u;
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    double c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) c[k] = sc.real(kSlotC + 3 * k + j);
    const int32_t m = imax(imax(hi_abs(c[0]), hi_abs(c[1])), hi_abs(c[2]));
    ok = ok && in_range(m);
    const int E = group_exp(m);
#pragma unroll
    for (int k = 0; k < 3; ++k) sc.put(kSlotC + 3 * k + j, limb(to_fixed<61>(c[k], E)));
    sc.put_word(kWordT + j, E - 1022);
  }

  // ---- nodal values (real U 2^(eu_i - 59)): gradient rows G (row 3: the
  // pressure's; real G 2^(eG_i + t_j - 61)), sums S and W (as U) ----
  Limb C[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[k][j] = sc.limb(kSlotC + 3 * k + j);
  uint32_t least = ~0u;
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    double u[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) u[a] = sc.real(kSlotU + 4 * i + a);
    const int32_t m = imax(imax(hi_abs(u[0]), hi_abs(u[1])), imax(hi_abs(u[2]), hi_abs(u[3])));
    ok = ok && in_range(m);
    const int E = group_exp(m);
    int64_t U[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) U[a] = to_fixed<59>(u[a], E);
    const int64_t S = (U[0] + U[1]) + (U[2] + U[3]);
    sc.put(kSlotS + i, S);
    sc.put_word(kWordEu + i, E - 1022);
    const int64_t D[3] = {U[1] - U[0], U[2] - U[0], U[3] - U[0]};
    const int sh = norm_shift64(D[0], D[1], D[2]);
    Limb Dl[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) Dl[k] = limb(shl(D[k], sh & 63));
    int64_t g[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) g[j] = dot3x<2>(Dl[0], C[0][j], Dl[1], C[1][j], Dl[2], C[2][j]);
    const int n = norm_shift(mag(g[0]) | mag(g[1]) | mag(g[2]));
    least = umin(least, umin(umin(mag(g[0]), mag(g[1])), mag(g[2])));
#pragma unroll
    for (int j = 0; j < 3; ++j) sc.put(kSlotG + 3 * i + j, shl(g[j], n));
    sc.put_word(kWordEg + i, (sh < 0 ? kZeroExp : E - 1021 - sh) + 2 - n);
    if (i < 3) {
      const int64_t bS = beta_sum(S);
#pragma unroll
      for (int a = 0; a < 4; ++a) sc.put(kSlotU + 4 * i + a, U[a] + bS);
    }
  }
  int t[3], eu[3], eG[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    t[j] = sc.word(kWordT + j);
    eu[j] = sc.word(kWordEu + j);
    eG[j] = sc.word(kWordEg + j);
  }
  const int egp = sc.word(kWordEg + 3);
  const int tmax = imax(t[0], imax(t[1], t[2]));
  ok = aligned_rows(sc, kSlotG, 4, 0, eu, t, tmax, least) && ok;
  if (!ok) return false;

  // ---- viscosity: a1 = -mu_eff / (6 detJ), real a1 2^(ea1 - 60) ----
  int einv;
  const Limb inv = limb(scalar_fixed(inv_det, einv));
  double mu_eff = P.P.mu;
  Limb a1l = P.a1.m;
  int ea1 = P.a1.e + einv;
  if constexpr (VREMAN) {
    double g[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) g[i][j] = to_double(sc.get(kSlotG + 3 * i + j), eG[i] + t[j] - 1);
    double vA, vphi, vscale;
    bool active = false;
    vreman_viscosity(g, rh, P, vA, vphi, vscale, mu_eff, active);
    if (active) {
      int em;
      const Limb mm = limb(scalar_fixed(mu_eff, em));
      // -mu_eff / 6 = -(2/3) 2^-2 mu_eff, as 2^(.. - 61)
      a1l = limb(mul8(mm, nsrhs::fixed::limb(-kTwoThirds61)) * 2);
      ea1 = em - 2 + einv;
    }
  }
  const int64_t a1 = mul8(inv, a1l);
  const double k1 = (VREMAN ? P.P.c1 * mu_eff : P.c1mu) * (rh * rh);

  // ---- Gauss points ----
  const int eum = imax(eu[0], imax(eu[1], eu[2]));
  const int kap = imax(eu[0] + t[0], imax(eu[1] + t[1], eu[2] + t[2]));
  int theta = -32768;
  const double k2 = (TAUE ? P.k2 : P.k2a) * rh;
  int64_t tme = 0;  // the per-element tau
  int ete = 0;
  double stau = 0.0;
  if constexpr (TAUE) {
    // |S / 4|^2
    const double sm = velocity_norm2(sc.get(kSlotS) >> 1, sc.get(kSlotS + 1) >> 1,
                                     sc.get(kSlotS + 2) >> 1, eu, eum) * 0.25;
    const double tau = M::rcp(fmac(k2, M::sqrt_(sm), k1));
    tme = scalar_fixed(tau, ete);
    stau = 4.0 * tau;
  }
  if constexpr (!TAUE) {
    // |W_g|^2 one after the other, then the four FP64 chains of tau side by
    // side (in the slots of tau W~ that the loop below fills last)
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      const double s = velocity_norm2(sc.get(kSlotU + g), sc.get(kSlotU + 4 + g),
                                      sc.get(kSlotU + 8 + g), eu, eum);
      sc.put_real(kSlotX + 8 + g, s);
    }
    double tau[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) tau[g] = M::rcp(fmac(k2, M::sqrt_(sc.real(kSlotX + 8 + g)), k1));
#pragma unroll
    for (int g = 0; g < 4; ++g) sc.put_real(kSlotX + 8 + g, tau[g]);
    stau = (tau[0] + tau[1]) + (tau[2] + tau[3]);
  }
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    int64_t w[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) w[i] = sc.get(kSlotU + 4 * i + g);
    int et = ete;
    int64_t tm = tme;
    if constexpr (!TAUE) tm = scalar_fixed(sc.real(kSlotX + 8 + g), et);
    const Limb tl = limb(tm);
    // W~, real 2^(kap - t_j - 59)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      w[j] = shr(w[j], kap - (eu[j] + t[j]));
      sc.put(kSlotWt + 4 * j + g, limb(w[j]));
    }
    // tau W~ from the normalised W~, real 2^(et - n + kap - t_j - 58)
    const int n = norm_shift(mag(w[0]) | mag(w[1]) | mag(w[2]));
    sc.put_word(kWordX + g, et - n);
    theta = imax(theta, et - n);
#pragma unroll
    for (int j = 0; j < 3; ++j) sc.put(kSlotX + 3 * g + j, mul8(tl, limb(shl(w[j], n))));
  }
  // T = sum tau W~, Q = sum tau W~ W~^T; (1 - beta) S = beta sum_a W_a
  // (u_a + S = W_a + (1 - beta) S)
  Limb Qp[6], sT[3], St[3];
  int eP, eT;
  {
    int64_t Tc[3] = {0, 0, 0}, V[3] = {0, 0, 0};
    Acc q[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) q[k] = acc_start();
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      const int k = theta - sc.word(kWordX + g);
      Limb v[3], w[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int64_t y = shr(sc.get(kSlotX + 3 * g + j), k);  // < 2^60, real 2^(theta + kap - t_j - 58)
        Tc[j] += y;
        v[j] = limb(y);
        w[j] = sc.limb(kSlotWt + 4 * j + g);
        V[j] += whole(w[j]);
      }
      mac(q[0], v[0], w[0]);
      mac(q[1], v[1], w[1]);
      mac(q[2], v[2], w[2]);
      mac(q[3], v[0], w[1]);
      mac(q[4], v[0], w[2]);
      mac(q[5], v[1], w[2]);
    }
    gauss_matrices(q, Tc, theta, kap, inv, einv, a1, ea1, t, tmax, P, Qp, eP, sT, eT);
#pragma unroll
    for (int j = 0; j < 3; ++j) St[j] = limb(beta_sum_wide(V[j]));
  }
  // psum / 24 = pb 2^(epb - 58): S is in units 2^(eu - 59), pb = S / 6
  const int64_t pb = mulx<1>(limb(sc.get(kSlotS + 3)), nsrhs::fixed::limb(kTwoThirds61));
  const int epb = sc.word(kWordEu + 3) - 3;

  // ---- rows 0..2: momentum, row 3: continuity ----
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    // F_a,i = base + sum_j K_j C_a,j (C_0 = -(C_1 + C_2 + C_3)) + sum_j H_j W~_a,j
    Limb Kl[3], Hl[3];
    int64_t base;
    int e;
    if (i < 3) {
      const int eg = sc.word(kWordEg + i), ti = sc.word(kWordT + i);
      const int e1 = eg + eP, e3 = egp + ti + eT, e5 = epb + ti, eh = P.m120.e + eg + kap;
      int eF = imax(imax(e1, e3), imax(e5, eh));
      Acc pp[3];
      int e4 = 0;
      if constexpr (SKEW) {
        e4 = P.r48.e + sc.word(kWordEu + i) + kap + 4;
        eF = imax(eF, e4);
#pragma unroll
        for (int j = 0; j < 3; ++j) pp[j] = accx_start<1>();
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
          const Limb w = limb(sc.get(kSlotU + 4 * i + g));
#pragma unroll
          for (int j = 0; j < 3; ++j) macx<1>(pp[j], w, sc.limb(kSlotWt + 4 * j + g));
        }
      }
      // K_ij = sum_k G_ik Qp_kj + gp_i sT_j + pb delta_ij, aligned through the
      // factors G_i and gp_i; real K 2^(eF - 58 - t_j), |K| < 2^61
      Limb Gs[3];
      int64_t K[3], H[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int64_t g = sc.get(kSlotG + 3 * i + j);
        Gs[j] = limb(shr(g, eF - e1));
        H[j] = shr(mul8(P.m120.m, limb(g)), eF - eh);
      }
      const Limb gpi = limb(shr(sc.get(kSlotG + 9 + i), eF - e3));
      const int64_t pbi = shr(pb, eF - e5);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Acc s = accx_start<1>(i == j ? pbi : 0);
        macx<1>(s, Gs[0], Qp[j == 0 ? 0 : j == 1 ? 3 : 4]);
        macx<1>(s, Gs[1], Qp[j == 0 ? 3 : j == 1 ? 1 : 5]);
        macx<1>(s, Gs[2], Qp[j == 0 ? 4 : j == 1 ? 5 : 2]);
        macx<1>(s, gpi, sT[j]);
        K[j] = finx<1>(s);
        if constexpr (SKEW) K[j] += shr(mulx<3>(P.r48.m, limb(finx<1>(pp[j]))), eF - e4);
      }
      const int n = norm_shift(mag(K[0]) | mag(K[1]) | mag(K[2]) | mag(H[0]) | mag(H[1]) |
                               mag(H[2]));
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Kl[j] = limb(shl(K[j], n));
        Hl[j] = limb(shl(H[j], n));
      }
      base = dot3(Hl[0], St[0], Hl[1], St[1], Hl[2], St[2]);
      e = eF - n + 5;
    } else {
      // F_a3 = -tr G / 24 + sum_j c_aj (sum_k sT_k G_jk - s24 stau gp_j)
      int es;
      const int64_t sm = scalar_fixed(stau, es);
      const Limb sg = limb(mul8(limb(mul8(inv, nsrhs::fixed::limb(-kTwoThirds61))), limb(sm * 2)));
      e = trace_row(sc, kSlotG, kSlotG + 9, kWordEg, kWordT, eG, t, tmax, sT, eT, sg,
                    einv - 4 + es + egp, -kTwoThirds61 / 2, kSlotX, Kl, base);
    }
    int64_t y[4];
    y[0] = base;
#pragma unroll
    for (int a = 1; a < 4; ++a) {
      y[a] = dot3(Kl[0], C[a - 1][0], Kl[1], C[a - 1][1], Kl[2], C[a - 1][2]);
      y[0] -= y[a];
      y[a] += base;
    }
    double f[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (i < 3)
        y[a] = dot3(Hl[0], sc.limb(kSlotWt + a), Hl[1], sc.limb(kSlotWt + 4 + a), Hl[2],
                    sc.limb(kSlotWt + 8 + a), y[a]);
      f[a] = to_double(y[a], e);
    }
    out(i, f);
  }
  return true;
}

// ---- host side ----

// x = m 2^(e - B), 2^(B - 1) <= |m| <= 2^B. x in long double (64 bits or
// more): a constant rounded to 53 bits would put the same relative error on
// every element.
inline Scalar make_scalar(long double x, int B) {
  Scalar s;
  s.m = {0, 0};
  s.e = kZeroExp;
  if (x != 0.0L) {
    const long double f = std::frexp(x, &s.e);  // 0.5 <= |f| < 1
    const int64_t m = std::llround(std::ldexp(f, B));
    s.m = {(int32_t)((m >> 32) + (int64_t)((uint32_t)m >> 31)), (int32_t)(uint32_t)m};
  }
  return s;
}

inline FixedParams make_fixed_params(const ElemParams<double>& P, bool skew) {
  const long double rho = P.rho, alpha = 1.0L / std::sqrt(5.0L);
  FixedParams q;
  q.P = P;
  q.c1mu = P.c1 * P.mu;
  q.k2 = P.c2 * P.rho;
  q.k2a = (double)(P.c2 * rho * alpha);
  q.rhoc = P.rho * P.c_vreman;
  q.a2 = make_scalar(-(rho * rho) / 120.0L, 61);  // alpha^2 = 1/5
  q.a1 = make_scalar(-(long double)P.mu / 6.0L, 61);
  q.b4 = make_scalar(-rho * alpha / 24.0L, 61);
  q.m120 = make_scalar(-rho / (skew ? 240.0L : 120.0L), 60);
  q.r48 = make_scalar(rho / 240.0L, 60);
  q.in_range = true;
  for (const double x : {P.rho, P.mu, P.c_vreman, P.c1, P.c2})
    q.in_range = q.in_range && (x == 0.0 || (x >= 0x1p-60 && x <= 0x1p60));
  return q;
}

}  // namespace fixed
}  // namespace nsrhs
