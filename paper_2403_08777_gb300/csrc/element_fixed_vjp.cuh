// The reverse sweep of element.cuh (element_vjp) split over the integer and
// the FP64 pipe; notation and scaling as in element_fixed.cuh.
//
// Integer pipe: gradient rows of the velocities, the pressure (G, gp) and the
// cotangent (Om = sum_a w_a c_a^T, cw), the Gauss point sums T and Q, the
// contractions G^T Om, the rows of Gb and their products with the cofactor
// vectors. They are the bulk of the products, and the rows of Gb and gpb have
// exactly the form of the forward's momentum and continuity rows.
// FP64 pipe: tau at the Gauss points, and the reverse sweep there with the
// eddy viscosity, the skew-symmetric term or the per-element tau. Without
// these the sweep has integer operands only, and an FP64 instruction takes its
// pipe 64 clocks, so it runs on the integer pipe as well: 256^3 52.2 -> 46.3
// ms (48.3 with the tau term's velocity at full width). Its terms mix the
// scaling of gradients and of velocities; each is normalised by itself, per
// Gauss point and component, before two meet.
#pragma once

#include "element_fixed.cuh"

namespace nsrhs {
namespace fixed {

// Slots of element_vjp_fixed, laid over one another so that 12 warps share
// an SM. U: velocities, component i of node a at kVjpU + 4 i + a; then W
// and u, aligned. X: cofactors (input c_k,j at kVjpC + 3 (k - 1) + j, then
// limbs); then the contractions for the Gauss points, tau and k2/|u_g|, and the
// Gauss points' gradients. W: the cotangent, component i of node a at kVjpW +
// 4 i + a; the slots of its component 3 end as a row's four sums. R: gradient
// rows of u, v, w, p and of the cotangent; the pressure's input values lie in
// the last four until its row is made, the pressure's row ends as scratch.
enum : int { kVjpU = 0, kVjpX = 12, kVjpC = kVjpX + 3, kVjpW = 24, kVjpR = 40, kVjpSlots = 64 };
enum : int { kVjpP = kVjpR + 20, kVjpY = kVjpW + 12, kVjpK = kVjpR + 9 };
enum : int { kVjpT = 0, kVjpEu = 3, kVjpEg = 11, kVjpXg = 19, kVjpWords = 31 };

// raw(i, a): component i of the velocity at node a as the caller's double.
template <int FLAGS, int THREADS, class Raw, class Out>
__device__ __forceinline__ bool element_vjp_fixed(const Scratch<THREADS>& sc, double inv_det,
                                                  double rh, const FixedParams& P,
                                                  const Raw& raw, const Out& out) {
  using M = MathOps<double>;
  constexpr bool VREMAN = (FLAGS & kVreman) != 0;
  constexpr bool SKEW = (FLAGS & kSkew) != 0;
  constexpr bool TAUE = (FLAGS & kTauElem) != 0;
  // the reverse sweep at the Gauss points on the integer pipe too
  constexpr bool INT = FLAGS == 0;
  // ---- cofactor vectors: real C 2^(t_j - 61) ----
  bool ok = (uint32_t)((hi_word(inv_det) >> 20) - 723) <= 600u &&
            (uint32_t)((hi_word(rh) >> 20) - 823) <= 400u;
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    double c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) c[k] = sc.real(kVjpC + 3 * k + j);
    const int32_t m = imax(imax(hi_abs(c[0]), hi_abs(c[1])), hi_abs(c[2]));
    ok = ok && in_range(m);
    const int E = group_exp(m);
#pragma unroll
    for (int k = 0; k < 3; ++k) sc.put(kVjpC + 3 * k + j, limb(to_fixed<61>(c[k], E)));
    sc.put_word(kVjpT + j, E - 1022);
  }
  Limb C[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[k][j] = sc.limb(kVjpC + 3 * k + j);

  // ---- nodal values of u, v, w, p and the cotangent (real U 2^(e_i - 59)):
  // gradient rows (real R 2^(eg_i + t_j - 61)), W of the velocities ----
  uint32_t least = ~0u;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    const int at = i < 3 ? kVjpU + 4 * i : i == 3 ? kVjpP : kVjpW + 4 * (i - 4);
    double u[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) u[a] = sc.real(at + a);
    const int32_t m = imax(imax(hi_abs(u[0]), hi_abs(u[1])), imax(hi_abs(u[2]), hi_abs(u[3])));
    ok = ok && in_range(m);
    const int E = group_exp(m);
    int64_t U[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) U[a] = to_fixed<59>(u[a], E);
    sc.put_word(kVjpEu + i, E - 1022);
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
    for (int j = 0; j < 3; ++j) sc.put(kVjpR + 3 * i + j, shl(g[j], n));
    sc.put_word(kVjpEg + i, (sh < 0 ? kZeroExp : E - 1021 - sh) + 2 - n);
    if (i < 3) {
      const int64_t bS = beta_sum((U[0] + U[1]) + (U[2] + U[3]));
#pragma unroll
      for (int a = 0; a < 4; ++a) sc.put(at + a, U[a] + bS);
    } else if (i > 3) {
      // w_a + sum_b w_b: both uses of the cotangent below take it with the sum,
      // sum_a w_a (u_a + S) = sum_a (w_a + sum_b w_b) u_a
      const int64_t s = (U[0] + U[1]) + (U[2] + U[3]);
#pragma unroll
      for (int a = 0; a < 4; ++a) sc.put(at + a, U[a] + s);
    }
  }
  int t[3], eu[3], eG[3], eO[3], ew[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    t[j] = sc.word(kVjpT + j);
    eu[j] = sc.word(kVjpEu + j);
    ew[j] = sc.word(kVjpEu + 4 + j);
    eG[j] = sc.word(kVjpEg + j);
    eO[j] = sc.word(kVjpEg + 4 + j);
  }
  const int egp = sc.word(kVjpEg + 3), ecw = sc.word(kVjpEg + 7);
  const int tmax = imax(t[0], imax(t[1], t[2]));
  ok = aligned_rows(sc, kVjpR, 8, 4, eu, t, tmax, least) && ok;
  if (!ok) return false;
  const int eum = imax(eu[0], imax(eu[1], eu[2]));
  const int kap = imax(eu[0] + t[0], imax(eu[1] + t[1], eu[2] + t[2]));
  auto row = [&](int i, int j) { return sc.get(kVjpR + 3 * i + j); };

  // ---- contractions for the reverse sweep at the Gauss points ----
  const double s24 = inv_det * (1.0 / 24.0);
  int einv;
  const Limb inv = limb(scalar_fixed(inv_det, einv));
  double mub = 0.0;   // mu_eff-bar (used with the eddy viscosity)
  double Qh[3][3], Tb[3], staub;
  // INT: alpha^2 Qh, with W~ in units 2^(eM + t_j - 60) (see below), alpha Tb in
  // units 2^(eA + t_j - 60), staub in units 2^(eB - 56)
  Limb Mq[6];
  int64_t A[3], st;
  int eM = 0, eA = 0, eB = 0;
  {
    uint32_t mx = 0, ma = 0;  // magnitudes of the two contractions
    int ex = 0, ea = 0;
    // Qh = (a2 / 2) (G^T Om + Om^T G): the component index aligned through G
    {
      const int e[3] = {eG[0] + eO[0], eG[1] + eO[1], eG[2] + eO[2]};
      const int m = imax(e[0], imax(e[1], e[2]));
      ex = m;
#pragma unroll 1
      for (int q = 0; q < 6; ++q) {  // entries 00 11 22 01 02 12
        const int j = q < 3 ? q : q == 5 ? 1 : 0, k = q < 3 ? q : q == 3 ? 1 : 2;
        Limb gj[3], gk[3], oj[3], ok_[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          gj[i] = limb(shr(row(i, j), m - e[i]));
          gk[i] = limb(shr(row(i, k), m - e[i]));
          oj[i] = limb(row(4 + i, j));
          ok_[i] = limb(row(4 + i, k));
        }
        // real 2^(m + t_j + t_k - 59), twice Qh / a2
        const int64_t x = dot3x<1>(gj[0], ok_[0], gj[1], ok_[1], gj[2], ok_[2]) +
                          dot3x<1>(gk[0], oj[0], gk[1], oj[1], gk[2], oj[2]);
        if constexpr (INT) {
          mx |= mag(x >> 1);
          sc.put(kVjpX + q, x >> 1);
        } else {
          sc.put_real(kVjpX + q, to_double(x, m + sc.word(kVjpT + j) + sc.word(kVjpT + k)));
        }
      }
    }
    // Tb = b4 (Om^T gp + G^T cw), staub = -s24 cw . gp
    {
      int m = egp + eO[0] + t[0];
#pragma unroll
      for (int i = 0; i < 3; ++i)
        m = imax(m, imax(egp + eO[i] + t[i], ecw + eG[i] + t[i]));
      ea = m;
      Limb a[3], b[3], d[3], f[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int64_t gp = row(3, i), cw = row(7, i);
        a[i] = limb(shr(gp, m - (egp + eO[i] + t[i])));
        b[i] = limb(shr(cw, m - (ecw + eG[i] + t[i])));
        d[i] = limb(shr(cw, 2 * (tmax - t[i])));
        f[i] = limb(gp);
      }
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        const int64_t x =
            dot3x<1>(a[0], limb(row(4, j)), a[1], limb(row(5, j)), a[2], limb(row(6, j))) +
            dot3x<1>(b[0], limb(row(0, j)), b[1], limb(row(1, j)), b[2], limb(row(2, j)));
        if constexpr (INT) {
          ma |= mag(x >> 1);
          sc.put(kVjpX + 6 + j, x >> 1);
        } else {
          sc.put_real(kVjpX + 6 + j, to_double(x, m + sc.word(kVjpT + j) + 1));
        }
      }
      const int64_t x = dot3x<1>(d[0], f[0], d[1], f[1], d[2], f[2]);
      if constexpr (INT)
        st = mul8(limb(mul8(inv, nsrhs::fixed::limb(-kTwoThirds61))), limb(x));
      else
        staub = -s24 * to_double(x, ecw + egp + 2 * tmax + 1);
    }
    if constexpr (INT) {
      const int nx = norm_shift(mx), na = norm_shift(ma);
      const Limb a2 = limb(mul8(inv, P.a2.m)), b4 = limb(mul8(inv, P.b4.m));
      eM = P.a2.e + einv + ex + kap + 4 - nx;
      eA = P.b4.e + einv + ea + 3 - na;
#pragma unroll
      for (int q = 0; q < 6; ++q) Mq[q] = limb(mul8(a2, limb(shl(sc.get(kVjpX + q), nx))));
#pragma unroll
      for (int j = 0; j < 3; ++j) A[j] = mul8(b4, limb(shl(sc.get(kVjpX + 6 + j), na)));
      const int ns = norm_shift(mag(st));
      eB = einv + ecw + egp + 2 * tmax - 6 - ns;
      st = shl(st, ns);
    } else {
      double x[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) x[q] = sc.real(kVjpX + q);
      if constexpr (VREMAN) mub = -4.0 * s24 * ((x[0] + x[1]) + x[2]);
      const double a2 = s24 * -(P.P.rho * P.P.rho), b4 = s24 * -P.P.rho;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Qh[j][j] = a2 * x[j];
        Tb[j] = b4 * sc.real(kVjpX + 6 + j);
      }
      Qh[0][1] = Qh[1][0] = a2 * x[3];
      Qh[0][2] = Qh[2][0] = a2 * x[4];
      Qh[1][2] = Qh[2][1] = a2 * x[5];
    }
  }

  // ---- viscosity ----
  double mu_eff = P.P.mu;
  double vA = 0.0, vphi = 0.0, vscale = 0.0;
  bool vactive = false;
  if constexpr (VREMAN) {
    double g[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) g[i][j] = to_double(row(i, j), eG[i] + t[j] - 1);
    vreman_viscosity(g, rh, P, vA, vphi, vscale, mu_eff, vactive);
  }
  const double rh2 = rh * rh;
  const double k1 = (VREMAN ? P.P.c1 * mu_eff : P.c1mu) * rh2;

  double stau = 0.0, tau_e = 0.0, yr_e = 0.0;
  double S[3] = {0.0, 0.0, 0.0};  // sum of the nodal velocities
  const double k2 = P.k2 * rh;
  int ete = 0;
  int64_t tme = 0;
  if constexpr (!INT) {
#pragma unroll
    for (int i = 0; i < 3; ++i) S[i] = (raw(i, 0) + raw(i, 1)) + (raw(i, 2) + raw(i, 3));
  }
  if constexpr (TAUE) {
    const double sm = fmac(S[2], S[2], fmac(S[1], S[1], S[0] * S[0])) * 0.0625;
    yr_e = M::rsqrt_(sm);
    tau_e = M::rcp(fmac(k2, sm * yr_e, k1));
    stau = 4.0 * tau_e;
    tme = scalar_fixed(tau_e, ete);
  }

  // ---- per Gauss point: tau_g and k2 / |u_g|, the normalisation of W~ ----
  const double k2a = P.k2a * rh;
  int theta = -32768;
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    int64_t w[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) w[j] = sc.get(kVjpU + 4 * j + g);
    int et = ete;
    if constexpr (!TAUE) {
      const double s = velocity_norm2(w[0], w[1], w[2], eu, eum);  // |u_g|^2 / alpha^2
      const double y = k2a * M::rsqrt_(s);                         // alpha^2 k2 / |u_g|
      const double tau = M::rcp(fmac(y, s, k1));
      sc.put_real(kVjpX + 3 * g, tau);
      sc.put_real(kVjpX + 3 * g + 1, y);
      stau += tau;
      et = scalar_exp(tau);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) w[j] = shr(w[j], kap - (eu[j] + t[j]));
    const int n = norm_shift(mag(w[0]) | mag(w[1]) | mag(w[2]));
    sc.put_word(kVjpXg + 3 * g, n);
    theta = imax(theta, et - n);
  }

  // ---- T, Q; Qp = a2 Q + a1 I, sT = b4 T ----
  Limb Qp[6], sT[3];
  int eP, eT;
  {
    int64_t Tc[3] = {0, 0, 0}, V[3] = {0, 0, 0};
    Acc q[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) q[k] = acc_start();
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      // tau W~ from the normalised W~, real 2^(et - n + kap - t_j - 58)
      int et = ete;
      int64_t tm = tme;
      if constexpr (!TAUE) tm = scalar_fixed(sc.real(kVjpX + 3 * g), et);
      const Limb tl = limb(tm);
      const int n = sc.word(kVjpXg + 3 * g), k = theta - (et - n);
      Limb v[3], w[3], wn[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int64_t x = shr(sc.get(kVjpU + 4 * j + g), kap - (eu[j] + t[j]));
        w[j] = limb(x);
        wn[j] = limb(shl(x, n));
        const int64_t y = shr(mul8(tl, wn[j]), k);
        Tc[j] += y;
        v[j] = limb(y);
        V[j] += x;
      }
      mac(q[0], v[0], w[0]);
      mac(q[1], v[1], w[1]);
      mac(q[2], v[2], w[2]);
      mac(q[3], v[0], w[1]);
      mac(q[4], v[0], w[2]);
      mac(q[5], v[1], w[2]);
      if constexpr (INT) {
        // alpha u_g-bar = tau (alpha Tb + 2 N) + alpha^2 sc W, N = alpha^2 Qh W,
        // alpha^2 sc = (alpha^2 k2 / |u_g|) (-tau^2) (staub + W . (alpha Tb + N))
        int64_t N[3], Y[3];
        N[0] = dot3x<3>(Mq[0], wn[0], Mq[3], wn[1], Mq[4], wn[2]);
        N[1] = dot3x<3>(Mq[3], wn[0], Mq[1], wn[1], Mq[5], wn[2]);
        N[2] = dot3x<3>(Mq[4], wn[0], Mq[5], wn[1], Mq[2], wn[2]);
        int eY = imax(eM - n, eA) + 3;
        const int dN = eY - (eM - n), dA = eY - eA;
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          N[i] = shr(N[i], dN);
          Y[i] = shr(A[i], dA) + N[i];
          m |= mag(Y[i]) | mag(N[i]);
        }
        const int nY = norm_shift(m) - 1;
        eY -= nY;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          N[i] = shl(Y[i] + N[i], nY);
          Y[i] = shl(Y[i], nY);
        }
        const int eD = eY + kap - n, eb = imax(eD, eB) + 1;
        const int64_t tb =
            shr(dot3x<1>(limb(Y[0]), wn[0], limb(Y[1]), wn[1], limb(Y[2]), wn[2]), eb - eD) +
            shr(st, eb - eB);
        const int nb = norm_shift(mag(tb));
        int ey;
        const double yd = sc.real(kVjpX + 3 * g + 1);
        int64_t ym = scalar_fixed(yd, ey);
        if (yd == 0.0) ym = 0;  // at rest
        const Limb ty = limb(mul8(limb(mul8(tl, limb(tm * 2))), limb(ym * 2)));
        const int64_t sw = -mul8(ty, limb(shl(tb, nb)));
        const int ns = norm_shift(mag(sw)) - 1;
        const Limb s2 = limb(shl(sw, ns));
        const int es = 2 * et + ey + eb - nb + 6 - ns;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          // the last term takes W as it is, not the aligned W~, which has lost a
          // bit per factor 2 of the cell's flatness
          const int64_t u = sc.get(kVjpU + 4 * i + g);
          const int nu = norm_shift(mag(u));
          const int64_t x = mul8(tl, limb(N[i])), y = mul8(s2, limb(shl(u, nu)));
          const int nx = norm_shift(mag(x));
          const int ex = et + eY + t[i] - nx, ey = es + eu[i] - nu, e = imax(ex, ey) + 1;
          sc.put(kVjpX + 3 * g + i, shr(shl(x, nx), e - ex) + shr(y, e - ey));
          sc.put_word(kVjpXg + 3 * g + i, e);
        }
      }
    }
    Limb a1l = P.a1.m;
    int ea1 = P.a1.e + einv;
    if constexpr (VREMAN) {
      if (vactive) {
        int em;
        const Limb mm = limb(scalar_fixed(mu_eff, em));
        a1l = limb(mul8(mm, nsrhs::fixed::limb(-kTwoThirds61)) * 2);
        ea1 = em - 2 + einv;
      }
    }
    gauss_matrices(q, Tc, theta, kap, inv, einv, mul8(inv, a1l), ea1, t, tmax, P, Qp, eP, sT, eT);
    // from W~_a to u_a = W_a - QB sum_b W_b (the sum is S sqrt 5)
#pragma unroll
    for (int j = 0; j < 3; ++j) V[j] = qb_sum(V[j]);
#pragma unroll 1
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        sc.put(kVjpU + 4 * j + a,
               limb(shr(sc.get(kVjpU + 4 * j + a), kap - (eu[j] + t[j])) - V[j]));
    if constexpr (INT) {
      // (QA - QB) u_a-bar + QB sum_g u_g-bar, QB = alpha beta
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        int e[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) e[g] = sc.word(kVjpXg + 3 * g + i);
        // |x| < 2^59, so that |x + U| <= (1 + 4 beta) 2^59 < 2^60.2: every reader
        // of these slots takes numbers below 2^61
        const int m = imax(imax(e[0], e[1]), imax(e[2], e[3])) + 2;
        int64_t x[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) x[g] = shr(sc.get(kVjpX + 3 * g + i), m - e[g]);
        const int64_t U = beta_sum_wide((x[0] + x[1]) + (x[2] + x[3]));
#pragma unroll
        for (int g = 0; g < 4; ++g) sc.put(kVjpX + 3 * g + i, x[g] + U);
        sc.put_word(kVjpXg + i, m - 4);
      }
    }
  }

  // ---- FP64: reverse sweep at the Gauss points ----
  if constexpr (!INT) {
    double Os[3][3];
    if constexpr (SKEW) {
      const double r48 = P.P.rho * (1.0 / 48.0);
      double o[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) o[i][j] = to_double(row(4 + i, j), eO[i] + t[j] - 1);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) Os[i][j] = r48 * (o[i][j] + o[j][i]);
    }
    double bS[3], Usum[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 3; ++i) bS[i] = kQB * S[i];
    const double crh2 = P.P.c1 * rh2;
    double Sb[3] = {0.0, 0.0, 0.0};  // S-bar from the per-element tau
    if constexpr (TAUE) {
      // tau-bar = 4 staub + Tb . S + <Qbar, sum_g u_g u_g^T>
      double taub = fmac(4.0, staub, fmac(Tb[2], S[2], fmac(Tb[1], S[1], Tb[0] * S[0])));
#pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        double ug[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) ug[i] = fmac(kQA - kQB, raw(i, g), bS[i]);
#pragma unroll
        for (int i = 0; i < 3; ++i)
          taub = fmac(ug[i], fmac(Qh[i][2], ug[2], fmac(Qh[i][1], ug[1], Qh[i][0] * ug[0])), taub);
      }
      const double db = -(tau_e * tau_e) * taub;
      if constexpr (VREMAN) mub = fmac(crh2, db, mub);
      const double scl = (k2 * db) * (yr_e * 0.0625);
#pragma unroll
      for (int i = 0; i < 3; ++i) Sb[i] = fmac(tau_e, Tb[i], scl * S[i]);
    }
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      double ug[3], ub[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) ug[i] = fmac(kQA - kQB, raw(i, g), bS[i]);
      if constexpr (!TAUE) {
        const double tau = sc.real(kVjpX + 3 * g), kyr = sc.real(kVjpX + 3 * g + 1);
        double QT[3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
          QT[i] = fmac(Qh[i][2], ug[2], fmac(Qh[i][1], ug[1], fmac(Qh[i][0], ug[0], Tb[i])));
        const double taub = fmac(ug[2], QT[2], fmac(ug[1], QT[1], fmac(ug[0], QT[0], staub)));
        const double db = -(tau * tau) * taub;
        if constexpr (VREMAN) mub = fmac(crh2, db, mub);
        const double scl = 5.0 * kyr * db;  // alpha^2 = 1/5
#pragma unroll
        for (int i = 0; i < 3; ++i) ub[i] = fmac(tau, fmac(2.0, QT[i], -Tb[i]), scl * ug[i]);
      } else {
        const double te2 = 2.0 * tau_e;
#pragma unroll
        for (int i = 0; i < 3; ++i)
          ub[i] = te2 * fmac(Qh[i][2], ug[2], fmac(Qh[i][1], ug[1], Qh[i][0] * ug[0]));
      }
      if constexpr (SKEW) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
          ub[i] = fmac(Os[i][0], ug[0], fmac(Os[i][1], ug[1], fmac(Os[i][2], ug[2], ub[i])));
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        Usum[i] += ub[i];
        sc.put_real(kVjpX + 3 * g + i, ub[i]);
      }
    }
    // (QA - QB) u_a-bar + QB sum_g u_g-bar (+ the per-element tau's part)
#pragma unroll
    for (int i = 0; i < 3; ++i) Sb[i] = fmac(kQB, Usum[i], Sb[i]);
    double B[3][3];
    if constexpr (VREMAN) {
      if (vactive) vreman_gradient([&](int i, int j) { return to_double(row(i, j), eG[i] + t[j] - 1); },
                                   mub, vA, vphi, vscale, B);
    }
#pragma unroll 1
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        double x = fmac(kQA - kQB, sc.real(kVjpX + 3 * a + i), Sb[i]);
        if constexpr (VREMAN) {
          if (vactive) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              const int64_t c1 = whole(C[0][j]), c2 = whole(C[1][j]), c3 = whole(C[2][j]);
              x = fmac(B[i][j], to_double(a == 0 ? -(c1 + c2 + c3) : a == 1 ? c1 : a == 2 ? c2 : c3, t[j] - 1), x);
            }
          }
        }
        sc.put_real(kVjpX + 3 * a + i, x);
      }
  }

  // ---- rows 0..2: velocity gradient, row 3: pressure gradient ----
  // (as the rows of the forward, with Om, cw and -sum_a w_a3 / 24 in the place
  // of G, gp and psum / 24)
  int64_t pb;
  int epb;
  {
    int64_t s = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a) s += sc.get(kVjpW + 12 + a) >> 3;
    // s = (5/8) sum_a w_a3 < 2^60.4
    pb = mulx<3>(nsrhs::fixed::limb(-kEightFifteenths60), limb(s));
    epb = sc.word(kVjpEu + 7) - 3;
  }
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    Limb Kl[3], Hl[3];
    int64_t base;
    int e, nr = 0;
    if (i < 3) {
      const int eo = sc.word(kVjpEg + 4 + i), ti = sc.word(kVjpT + i), ewi = sc.word(kVjpEu + 4 + i);
      const int e1 = eo + eP, e3 = ecw + ti + eT, e5 = epb + ti, e6 = P.m120.e + ewi + kap + 4;
      int eF = imax(imax(e1, e3), imax(e5, e6));
      // Hm_ki = m120 G_ki, aligned over the components k
      const int eh = P.m120.e + ti;
#pragma unroll
      for (int k = 0; k < 3; ++k) eF = imax(eF, eh + eG[k] + ew[k]);
      // INT: the Gauss points' part of node a's gradient
      const int er = INT ? sc.word(kVjpXg + i) : 0;
      if constexpr (INT) eF = imax(eF, er);
      uint32_t mh = 0;
      // sum_a w_ai v_a, v_a = m120 (u_a + S)
      Acc wv[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) wv[j] = accx_start<1>();
#pragma unroll 1
      for (int a = 0; a < 4; ++a) {
        const Limb wl = limb(sc.get(kVjpW + 4 * i + a));
#pragma unroll
        for (int j = 0; j < 3; ++j) macx<1>(wv[j], wl, sc.limb(kVjpU + 4 * j + a));
        if constexpr (INT) mh |= mag(shr(sc.get(kVjpX + 3 * a + i), eF - er));
      }
      Limb Os[3];
      int64_t K[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) Os[j] = limb(shr(sc.get(kVjpR + 12 + 3 * i + j), eF - e1));
      const Limb cwi = limb(shr(sc.get(kVjpR + 21 + i), eF - e3));
      const int64_t pbi = shr(pb, eF - e5);
#pragma unroll 1
      for (int k = 0; k < 3; ++k) {
        const int64_t h = shr(mul8(P.m120.m, limb(sc.get(kVjpR + 3 * k + i))),
                              eF - (eh + sc.word(kVjpEg + k) + sc.word(kVjpEu + 4 + k)));
        mh |= mag(h);
        sc.put(kVjpK + k, h);
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Acc s = accx_start<1>(i == j ? pbi : 0);
        macx<1>(s, Os[0], Qp[j == 0 ? 0 : j == 1 ? 3 : 4]);
        macx<1>(s, Os[1], Qp[j == 0 ? 3 : j == 1 ? 1 : 5]);
        macx<1>(s, Os[2], Qp[j == 0 ? 4 : j == 1 ? 5 : 2]);
        macx<1>(s, cwi, sT[j]);
        K[j] = finx<1>(s) + shr(mulx<3>(P.m120.m, limb(finx<1>(wv[j]))), eF - e6);
      }
      const int n = norm_shift(mag(K[0]) | mag(K[1]) | mag(K[2]) | mh);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Kl[j] = limb(shl(K[j], n));
        Hl[j] = limb(shl(sc.get(kVjpK + j), n));
      }
      base = 0;
      nr = eF - n - er;
      e = eF - n + 5;
    } else {
      // tr Om / 24 + sum_j c_aj (sum_k sT_k Om_jk - s24 stau cw_j)
      int es;
      const int64_t sm = scalar_fixed(stau, es);
      const Limb sg = limb(mul8(limb(mul8(inv, nsrhs::fixed::limb(-kTwoThirds61))), limb(sm * 2)));
      e = trace_row(sc, kVjpR + 12, kVjpR + 21, kVjpEg + 4, kVjpT, eO, t, tmax, sT, eT, sg, einv - 4 + es + ecw,
                    kTwoThirds61 / 2, kVjpK, Kl, base);
    }
    int64_t y[4];
    y[0] = base;
#pragma unroll
    for (int a = 1; a < 4; ++a) {
      y[a] = dot3(Kl[0], C[a - 1][0], Kl[1], C[a - 1][1], Kl[2], C[a - 1][2]);
      y[0] -= y[a];
      y[a] += base;
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) sc.put(kVjpY + a, y[a]);
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
      int64_t z = sc.get(kVjpY + a);
      double x = 0.0;
      if (i < 3) {
        z = dot3(Hl[0], limb(sc.get(kVjpW + a)), Hl[1], limb(sc.get(kVjpW + 4 + a)), Hl[2],
                 limb(sc.get(kVjpW + 8 + a)), z);
        if constexpr (INT)
          z += nr < 0 ? shl(sc.get(kVjpX + 3 * a + i), -nr) : shr(sc.get(kVjpX + 3 * a + i), nr);
        else
          x = sc.real(kVjpX + 3 * a + i);
      }
      out(i, a, INT ? to_double(z, e) : to_double(z, e) + x);
    }
  }
  return true;
}

}  // namespace fixed
}  // namespace nsrhs
