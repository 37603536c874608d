// Host check of the block fixed-point arithmetic (csrc/fixed.cuh) and of the
// element routines built on it (csrc/element_fixed.cuh): the same sources,
// compiled with tests/flopcount/cuda_runtime.h in place of CUDA's.
//   primitives: conversions and products at the edges of their ranges, in
//     units of the last place they promise;
//   routines: errors against the element's weak form in long double, beside
//     the errors of the double-precision routine, norm-wise per component.
// Prints one line per check: "name value limit".
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <random>

#include "../../paper_2403_08777_gb300/csrc/element_fixed.cuh"
#include "../../paper_2403_08777_gb300/csrc/element_fixed_vjp.cuh"

using namespace nsrhs;
using fixed::limb;

// The element's right-hand side at the Gauss points, term by term, in long
// double (or complex long double, for derivatives by the complex step).
typedef long double ld;
static ld real(ld x) { return x; }
static ld real(const std::complex<ld>& x) { return x.real(); }
template <int FLAGS, class T>
static void reference(const double Xd[4][3], const T u[4][3], const T p[4], const ElemParams<double>& P,
                      T F[4][4]) {
  ld e[3][3], c[3][3], dn[4][3];
  for (int k = 0; k < 3; ++k)
    for (int d = 0; d < 3; ++d) e[k][d] = (ld)Xd[k + 1][d] - Xd[0][d];
  for (int k = 0; k < 3; ++k) {
    const ld *a = e[(k + 1) % 3], *b = e[(k + 2) % 3];
    c[k][0] = a[1] * b[2] - a[2] * b[1];
    c[k][1] = a[2] * b[0] - a[0] * b[2];
    c[k][2] = a[0] * b[1] - a[1] * b[0];
  }
  const ld det = e[0][0] * c[0][0] + e[0][1] * c[0][1] + e[0][2] * c[0][2];
  for (int j = 0; j < 3; ++j) {
    for (int k = 0; k < 3; ++k) dn[k + 1][j] = c[k][j] / det;
    dn[0][j] = -(dn[1][j] + dn[2][j] + dn[3][j]);
  }
  const ld h = std::cbrt(det), rho = P.rho, QA = (5 + 3 * std::sqrt((ld)5)) / 20, QB = (5 - std::sqrt((ld)5)) / 20;
  T G[3][3], gp[3], sum[3], mu = (ld)P.mu;
  for (int i = 0; i < 3; ++i) {
    sum[i] = u[0][i] + u[1][i] + u[2][i] + u[3][i];
    gp[i] = p[0] * dn[0][i] + p[1] * dn[1][i] + p[2] * dn[2][i] + p[3] * dn[3][i];
    for (int j = 0; j < 3; ++j)
      G[i][j] = u[0][i] * dn[0][j] + u[1][i] * dn[1][j] + u[2][i] * dn[2][j] + u[3][i] * dn[3][j];
  }
  if (FLAGS & kVreman) {
    T b[3][3], A = 0;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        b[i][j] = h * h * (G[i][0] * G[j][0] + G[i][1] * G[j][1] + G[i][2] * G[j][2]);
        A += G[i][j] * G[i][j];
      }
    const T B = b[0][0] * b[1][1] - b[0][1] * b[0][1] + b[0][0] * b[2][2] - b[0][2] * b[0][2] +
                b[1][1] * b[2][2] - b[1][2] * b[1][2];
    if (real(A) > 0 && real(B) > 0) mu += rho * (ld)P.c_vreman * std::sqrt(B / A);
  }
  auto tau_of = [&](const T v[3]) {
    const T s = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    const T n = real(s) > 0 ? std::sqrt(s) : T(0);
    return (ld)1 / ((ld)P.c1 * mu / (h * h) + (ld)P.c2 * rho * n / h);
  };
  const T mean[3] = {sum[0] / (ld)4, sum[1] / (ld)4, sum[2] / (ld)4};
  for (int a = 0; a < 4; ++a)
    for (int k = 0; k < 4; ++k) F[a][k] = 0;
  for (int g = 0; g < 4; ++g) {
    T ug[3], cv[3], r[3];
    for (int i = 0; i < 3; ++i) ug[i] = QB * sum[i] + (QA - QB) * u[g][i];
    const T pg = QB * (p[0] + p[1] + p[2] + p[3]) + (QA - QB) * p[g];
    for (int i = 0; i < 3; ++i) {
      cv[i] = ug[0] * G[i][0] + ug[1] * G[i][1] + ug[2] * G[i][2];
      r[i] = rho * cv[i] + gp[i];
    }
    const T tau = tau_of(FLAGS & kTauElem ? mean : ug);
    for (int a = 0; a < 4; ++a) {
      const ld N = a == g ? QA : QB, w = det / 24;
      const T un = ug[0] * dn[a][0] + ug[1] * dn[a][1] + ug[2] * dn[a][2];
      for (int i = 0; i < 3; ++i) {
        T f = FLAGS & kSkew ? -rho / 2 * (N * cv[i] - un * ug[i]) : -rho * N * cv[i];
        f += -mu * (dn[a][0] * G[i][0] + dn[a][1] * G[i][1] + dn[a][2] * G[i][2]) + pg * dn[a][i] -
             tau * rho * un * r[i];
        F[a][i] += w * f;
      }
      F[a][3] += w * (-N * (G[0][0] + G[1][1] + G[2][2]) -
                      tau * (dn[a][0] * r[0] + dn[a][1] * r[1] + dn[a][2] * r[2]));
    }
  }
}

static std::mt19937_64 rng(7);
static double uni(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }
static double normal() { return std::normal_distribution<double>()(rng); }
static void say(const char* name, int a, int b, double value, double limit) {
  std::printf("%s[%d,%d] %.17g %.17g\n", name, a, b, value, limit);
}

static void primitives() {
  // to_double: half a unit in the last place, for every position of the leading bit
  double worst = 0;
  auto conv = [&](int64_t x, int e) {
    const long double want = std::ldexp((long double)x, e - 60);
    const double got = fixed::to_double(x, e);
    if (x == 0)
      worst = std::max(worst, got == 0 ? 0.0 : 1e9);
    else
      worst = std::max(worst, (double)(std::fabs(got - want) / std::fabs(want)) * 0x1p53);
  };
  for (int b = 0; b < 63; ++b)
    for (int d = -3; d <= 3; ++d) conv((1ll << b) + d, -5), conv(-((1ll << b) + d), 9);
  for (int i = 0; i < 200000; ++i) conv((int64_t)rng() >> (1 + rng() % 63), (int)(rng() % 200) - 100);
  say("to_double", 0, 0, worst, 1.0 + 1e-9);
  // to_fixed: less than one unit of the group below the value's magnitude
  worst = 0;
  for (int i = 0; i < 200000; ++i) {
    const int E = 900 + (int)(rng() % 240);
    double x = std::ldexp(uni(0.5, 1), E - 1022 - (int)(rng() % 70)) * (rng() & 1 ? 1 : -1);
    if (i % 5 == 0) x = std::ldexp(1 - 0x1p-53, E - 1022) * (rng() & 1 ? 1 : -1);
    const int64_t X = fixed::to_fixed<61>(x, E);
    worst = std::max(worst, (double)std::fabs((long double)X - std::ldexp((long double)x, 1022 + 61 - E)));
  }
  say("to_fixed", 0, 0, worst, 1.0);
  // products against 128-bit integers, mantissas of ones among the operands;
  // per product: the dropped l l' / 2^64 (1/4) and the truncation (1/2, 1 with mul8's 8)
  double e0 = 0, e1 = 0, e2 = 0, e3 = 0, e8 = 0, es = 0, ew = 0;
  for (int i = 0; i < 400000; ++i) {
    int64_t a = (int64_t)rng() >> (3 + rng() % 8), b = (int64_t)rng() >> (3 + rng() % 8);
    if (i % 7 == 0) a = (1ll << 61) - 1 - (int64_t)(rng() % 3);
    if (i % 11 == 0) b = -((1ll << 61) - (int64_t)(rng() % 3));
    if (i % 13 == 0) a = -(1ll << 61), b = 1ll << 61;
    const int64_t h = a >> 1;
    auto err = [](int64_t got, int64_t x, int64_t y, int s) {
      return (double)std::fabs((long double)got - std::ldexp((long double)x * (long double)y, s - 64));
    };
    e0 = std::max(e0, err(fixed::mul(limb(a), limb(b)), a, b, 0));
    e1 = std::max(e1, err(fixed::mulx<1>(limb(a), limb(b)), a, b, 1));
    e2 = std::max(e2, err(fixed::mulx<2>(limb(h), limb(b)), h, b, 2));
    e3 = std::max(e3, err(fixed::mulx<3>(limb(h), limb(b)), h, b, 3));
    e8 = std::max(e8, err(fixed::mul8(limb(h), limb(b)), h, b, 3));
    es = std::max(es, (double)std::fabs((long double)fixed::square3(limb(a), limb(b), limb(h)) -
                                        std::ldexp((long double)a * a + (long double)b * b +
                                                       (long double)h * h, -64)));
    ew = std::max(ew, fixed::whole(limb(a)) == a ? 0.0 : 1.0);
  }
  say("mul", 0, 0, e0, 0.25 + 1.0);
  say("mulx", 1, 0, e1, 0.5 + 1.0);
  say("mulx", 2, 0, e2, 1.0 + 1.0);
  say("mulx", 3, 0, e3, 2.0 + 1.0);
  say("mul8", 0, 0, e8, 2.0 + 8.0);
  say("square3", 0, 0, es, 0.75 + 2.0);
  say("whole", 0, 0, ew, 0.0);
}

// Element data. kind: 0 Taylor-Green + noise, 1 random vectors up to 10 (some
// with mantissas of ones), 2 flat cells (1 : 100), 3 nearly constant velocity
// with components of different size, 4 a velocity at one node only, 5 at rest.
struct Element {
  double X[4][3], u[4][3], p[4], w[4][4], c[3][3], inv, rh;
  ElemParams<double> P;
};
static Element make(int kind, int it) {
  Element q;
  static const int perm[6][3] = {{0, 1, 2}, {1, 2, 0}, {2, 0, 1}, {0, 2, 1}, {2, 1, 0}, {1, 0, 2}};
  const int t = (int)(rng() % 6);
  double l[4][3] = {};
  for (int s = 0; s < 3; ++s) {
    for (int d = 0; d < 3; ++d) l[s + 1][d] = l[s][d];
    l[s + 1][perm[t][s]] += 1;
  }
  if (t >= 3)
    for (int d = 0; d < 3; ++d) std::swap(l[1][d], l[2][d]);
  const double off[3] = {std::floor(uni(0, 64)), std::floor(uni(0, 64)), std::floor(uni(0, 64))};
  for (int a = 0; a < 4; ++a)
    for (int d = 0; d < 3; ++d)
      q.X[a][d] = (l[a][d] + off[d] + 0.12 * uni(-1, 1)) / 64 / (d == 2 && kind == 2 ? 100 : 1);
  for (int a = 0; a < 4; ++a) {
    const double T = 2 * M_PI, x = T * q.X[a][0], y = T * q.X[a][1], z = T * q.X[a][2];
    const double v[3] = {std::sin(x) * std::cos(y) * std::cos(z), -std::cos(x) * std::sin(y) * std::cos(z), 0};
    for (int i = 0; i < 3; ++i) {
      q.u[a][i] = v[i] + 1e-2 * normal();
      if (kind == 1) q.u[a][i] += uni(0, 10) * normal();
      if (kind == 1 && it % 4 == 0)
        q.u[a][i] = std::ldexp(1 - std::ldexp(1.0, -1 - (int)(rng() % 53)), (int)(rng() % 6) - 3) * (rng() & 1 ? 1 : -1);
      if (kind == 3) q.u[a][i] = i == 0 ? 10 + 1e-6 * normal() : (i == 1 ? 1e-5 : 1e-8) * normal();
      if (kind == 4) q.u[a][i] = a == it % 4 && i == 0 ? 1 : 0;
      if (kind == 5) q.u[a][i] = 0;
    }
    q.p[a] = uni(-1, 1);
    for (int k = 0; k < 4; ++k) q.w[a][k] = normal();
  }
  element_geometry<double, double>(q.X, q.c, q.inv, q.rh);
  q.P = {1.0, kind == 1 ? 1e-4 : 1e-2, 0.07, 4, 2};
  return q;
}

struct Keep {
  double (*F)[4];
  void operator()(int k, const double f[4]) const {
    for (int a = 0; a < 4; ++a) F[a][k] = f[a];
  }
  void operator()(int k, int a, double f) const { F[a][k] = f; }
};
static void stage(const Element& q, int64_t* slots) {
  for (int k = 0; k < 9; ++k) std::memcpy(slots + fixed::kSlotC + k, &q.c[k / 3][k % 3], 8);
  for (int a = 0; a < 4; ++a) {
    for (int i = 0; i < 3; ++i) std::memcpy(slots + fixed::kSlotU + 4 * i + a, &q.u[a][i], 8);
    std::memcpy(slots + fixed::kSlotU + 12 + a, &q.p[a], 8);
  }
}

template <int FLAGS>
static void routine(int kind, int n) {
  double e[4] = {}, d[4] = {}, norm[4] = {};
  int left = 0;
  for (int it = 0; it < n; ++it) {
    const Element q = make(kind, it);
    const auto FP = fixed::make_fixed_params(q.P, (FLAGS & kSkew) != 0);
    double F[4][4], G[4][4];
    element_rhs<double, FLAGS>(q.c, q.inv, q.rh, q.u, q.p, q.P, F);
    int64_t slots[128];
    int16_t words[32];
    stage(q, slots);
    if (!fixed::element_rhs_fixed<FLAGS, 1>({slots, words}, q.inv, q.rh, FP, Keep{G})) ++left;
    ld u[4][3], p[4], R[4][4];
    for (int a = 0; a < 4; ++a) {
      for (int i = 0; i < 3; ++i) u[a][i] = q.u[a][i];
      p[a] = q.p[a];
    }
    reference<FLAGS, ld>(q.X, u, p, q.P, R);
    for (int a = 0; a < 4; ++a)
      for (int k = 0; k < 4; ++k) {
        e[k] += std::pow((double)(G[a][k] - R[a][k]), 2);
        d[k] += std::pow((double)(F[a][k] - R[a][k]), 2);
        norm[k] += std::pow((double)R[a][k], 2);
      }
  }
  say("left", FLAGS, kind, left, 0);
  for (int k = 0; k < 4; ++k)
    if (norm[k] > 0)
      say(k < 3 ? "momentum" : "continuity", FLAGS, kind, std::sqrt(e[k] / norm[k]),
          1.1 * std::sqrt(d[k] / norm[k]));
}
// The reverse sweep against complex-step derivatives of the reference.
// With rest (kinds 4, 5), where the derivative of |u_g| is 0 by convention,
// against the FP64 routine: two results, each within the 4.2e-16 that kinds
// 0 to 3 allow.
template <int FLAGS>
static void adjoint(int kind, int n) {
  typedef std::complex<ld> cld;
  double e[4] = {}, d[4] = {}, norm[4] = {};
  int left = 0;
  for (int it = 0; it < n; ++it) {
    const Element q = make(kind, it);
    const auto FP = fixed::make_fixed_params(q.P, (FLAGS & kSkew) != 0);
    double gu[4][3], gp[4], G[4][4];
    element_vjp<double, FLAGS>(q.c, q.inv, q.rh, q.u, q.p, q.w, q.P, gu, gp);
    int64_t slots[128];
    int16_t words[32];
    for (int k = 0; k < 9; ++k) std::memcpy(slots + fixed::kVjpC + k, &q.c[k / 3][k % 3], 8);
    for (int a = 0; a < 4; ++a) {
      for (int i = 0; i < 3; ++i) std::memcpy(slots + fixed::kVjpU + 4 * i + a, &q.u[a][i], 8);
      std::memcpy(slots + fixed::kVjpP + a, &q.p[a], 8);
      for (int i = 0; i < 4; ++i) std::memcpy(slots + fixed::kVjpW + 4 * i + a, &q.w[a][i], 8);
    }
    if (!fixed::element_vjp_fixed<FLAGS, 1>({slots, words}, q.inv, q.rh, FP,
                                            [&](int i, int a) { return q.u[a][i]; }, Keep{G}))
      ++left;
    const ld step = 1e-30L;
    for (int b = 0; b < 4; ++b)
      for (int k = 0; k < 4; ++k) {
        cld u[4][3], p[4], F[4][4];
        for (int a = 0; a < 4; ++a) {
          for (int i = 0; i < 3; ++i) u[a][i] = cld(q.u[a][i], a == b && i == k ? step : 0);
          p[a] = cld(q.p[a], a == b && k == 3 ? step : 0);
        }
        reference<FLAGS, cld>(q.X, u, p, q.P, F);
        ld r = 0;
        for (int a = 0; a < 4; ++a)
          for (int i = 0; i < 4; ++i) r += q.w[a][i] * (F[a][i].imag() / step);
        const double mine = k < 3 ? gu[b][k] : gp[b];
        if (kind > 3) r = mine;
        e[k] += std::pow((double)(G[b][k] - r), 2);
        d[k] += std::pow((double)(mine - r), 2);
        norm[k] += std::pow((double)r, 2);
      }
  }
  say("left_vjp", FLAGS, kind, left, 0);
  for (int k = 0; k < 4; ++k)
    say(k < 3 ? "velocity_grad" : "pressure_grad", FLAGS, kind, std::sqrt(e[k] / norm[k]),
        kind > 3 ? 8.4e-16 : 1.1 * std::sqrt(d[k] / norm[k]));
}
template <int FLAGS>
static void routines(int n) {
  // the eddy viscosity of kinds 2 and 3 is ill-conditioned in any arithmetic
  for (int kind : {0, 1, 2, 3, 4, 5})
    if (!(FLAGS & kVreman) || kind < 2 || kind > 3) routine<FLAGS>(kind, n);
  for (int kind : {0, 1, 2, 3, 4, 5})
    if (!(FLAGS & kVreman) || kind < 2) adjoint<FLAGS>(kind, n / 4);
}

// Data outside the range leave the routine before it has written anything.
static void range() {
  struct Never {
    int* n;
    void operator()(int, const double*) const { ++*n; }
  };
  int bad = 0, calls = 0;
  const double values[] = {INFINITY, -INFINITY, NAN, 1e40, -1e40, 1e-40, 0x1p-1074, 1e300};
  for (const double x : values)
    for (int at = 0; at < 8; ++at) {
      Element q = make(0, 0);
      if (at < 3) for (int a = 0; a < 4; ++a) q.u[a][at] = a == 1 || std::fabs(x) < 1 ? x : q.u[a][at];
      if (at == 3) for (int a = 0; a < 4; ++a) q.p[a] = a == 2 || std::fabs(x) < 1 ? x : q.p[a];
      if (at > 3 && at < 7) for (int k = 0; k < 3; ++k) q.c[k][at - 4] = x;
      if (at == 7) q.inv = std::fabs(x) == 0x1p-1074 ? 1e-300 : x == 1e40 || x == -1e40 || x == 1e-40 ? INFINITY : x;
      if (x == 0x1p-1074 && at < 7) continue;  // subnormal data count as 0
      int64_t slots[128];
      int16_t words[32];
      stage(q, slots);
      const auto FP = fixed::make_fixed_params(q.P, false);
      if (fixed::element_rhs_fixed<0, 1>({slots, words}, q.inv, q.rh, FP, Never{&calls})) ++bad;
    }
  say("range", 0, 0, bad + calls, 0);
}

int main() {
  primitives();
  range();
  const int n = 4000;
  routines<0>(n);
  routines<kVreman>(n);
  routines<kSkew>(n);
  routines<kVreman | kSkew>(n);
  routines<kTauElem>(n);
  routines<kVreman | kSkew | kTauElem>(n);
  return 0;
}
