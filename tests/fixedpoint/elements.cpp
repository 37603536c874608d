// Host check of the fixed-point element routines over elements of many kinds,
// beside check.cpp, whose reference and helpers it uses: what the arithmetic
// relies on (NSRHS_FIXED_EXPECT: shift counts that are not negative, no bits
// lost at the top of a number, accumulators and results in range) holds in
// every element, and the results are those of the double-precision routines.
// Prints one line per check: "name value limit".
static long g_violations = 0;
#define NSRHS_FIXED_EXPECT(ok) (void)((ok) || ++g_violations)
#define main check_main
#include "check.cpp"
#undef main

struct Results {
  double rhs[4][4], vjp[4][4];  // [node][component]
};
template <int FLAGS>
static bool by_fixed(const Element& q, Results& r) {
  const auto FP = fixed::make_fixed_params(q.P, (FLAGS & kSkew) != 0);
  int64_t slots[128];
  int16_t words[64];
  stage(q, slots);
  if (!fixed::element_rhs_fixed<FLAGS, 1>({slots, words}, q.inv, q.rh, FP, Keep{r.rhs})) return false;
  for (int k = 0; k < 9; ++k) std::memcpy(slots + fixed::kVjpC + k, &q.c[k / 3][k % 3], 8);
  for (int a = 0; a < 4; ++a) {
    for (int i = 0; i < 3; ++i) std::memcpy(slots + fixed::kVjpU + 4 * i + a, &q.u[a][i], 8);
    std::memcpy(slots + fixed::kVjpP + a, &q.p[a], 8);
    for (int i = 0; i < 4; ++i) std::memcpy(slots + fixed::kVjpW + 4 * i + a, &q.w[a][i], 8);
  }
  return fixed::element_vjp_fixed<FLAGS, 1>({slots, words}, q.inv, q.rh, FP,
                                            [&](int i, int a) { return q.u[a][i]; }, Keep{r.vjp});
}
template <int FLAGS>
static void by_double(const Element& q, Results& r) {
  double gu[4][3], gp[4];
  element_rhs<double, FLAGS>(q.c, q.inv, q.rh, q.u, q.p, q.P, r.rhs);
  element_vjp<double, FLAGS>(q.c, q.inv, q.rh, q.u, q.p, q.w, q.P, gu, gp);
  for (int a = 0; a < 4; ++a) {
    for (int i = 0; i < 3; ++i) r.vjp[a][i] = gu[a][i];
    r.vjp[a][3] = gp[a];
  }
}

// Differences of two routines over many elements, norm-wise per component.
struct Sum {
  double d[8] = {}, n[8] = {};
  void add(const Results& x, const Results& ref) {
    for (int a = 0; a < 4; ++a)
      for (int k = 0; k < 4; ++k) {
        d[k] += std::pow(x.rhs[a][k] - ref.rhs[a][k], 2);
        n[k] += std::pow(ref.rhs[a][k], 2);
        d[4 + k] += std::pow(x.vjp[a][k] - ref.vjp[a][k], 2);
        n[4 + k] += std::pow(ref.vjp[a][k], 2);
      }
  }
  double worst() const {
    double w = 0;
    for (int k = 0; k < 8; ++k)
      if (n[k] > 0) w = std::max(w, std::sqrt(d[k] / n[k]));
    return w;
  }
};

// Low velocities: 0 nearly uniform, 1 at one node only (beside a no-slip
// wall), at the given cell Reynolds number, pressures of order 1.
static Element low_velocity(int kind, double reynolds, double mu, double flat) {
  Element q = make(0, 0);
  for (int a = 0; a < 4; ++a) q.X[a][2] /= flat;
  element_geometry<double, double>(q.X, q.c, q.inv, q.rh);
  const double U = reynolds * mu * 64, spread = std::pow(10.0, uni(-8, -1));
  const double dir[3] = {normal(), normal(), normal()};
  const int node = (int)(rng() % 4);
  for (int a = 0; a < 4; ++a)
    for (int i = 0; i < 3; ++i)
      q.u[a][i] = kind == 0 ? U * (dir[i] + spread * normal()) : a == node ? U * normal() : 0.0;
  q.P.mu = mu;
  return q;
}
// The library's tolerance for FP64 results, 1e-12 norm-wise.
template <int FLAGS>
static void low_velocities(int n) {
  for (const int kind : {0, 1})
    for (const double mu : {1e-4, 1e-2})
      for (const double flat : {1.0, 20.0}) {
        Sum s;
        int left = 0;
        g_violations = 0;
        for (int it = 0; it < n; ++it) {
          const Element q = low_velocity(kind, std::pow(10.0, uni(-2, 0.3)), mu, flat);
          Results x, ref;
          by_double<FLAGS>(q, ref);
          if (!by_fixed<FLAGS>(q, x)) ++left;
          else s.add(x, ref);
        }
        const int id = 100 * kind + 10 * (mu > 1e-3) + (flat > 1);
        say("low_velocity_expect", FLAGS, id, (double)g_violations, 0);
        say("low_velocity_left", FLAGS, id, left, 0);
        // the gradient of a velocity at one node has rank 1, where the eddy
        // viscosity is the square root of a rounding error in any arithmetic
        if (kind == 0 || !(FLAGS & kVreman)) say("low_velocity", FLAGS, id, s.worst(), 1e-12);
      }
}

// What the arithmetic relies on, for check.cpp's kinds of elements.
template <int FLAGS>
static void expectations(int n) {
  for (int kind = 0; kind < 6; ++kind) {
    g_violations = 0;
    for (int it = 0; it < n; ++it) {
      Results x;
      by_fixed<FLAGS>(make(kind, it), x);
    }
    say("expect", FLAGS, kind, (double)g_violations, 0);
  }
}

// A wall cell whose four Gauss points add up alike: their sum needs the last
// bit that a stored number has.
static void wall_cell() {
  Element q = {
      {{0.73412880520138168, 0.45151404638763065, 0.5609918590211681},
       {0.74820741898590692, 0.45335968290017303, 0.5620100571258726},
       {0.75128004838359452, 0.46875315366672304, 0.56210945379511901},
       {0.75012502088914668, 0.47061793926641393, 0.5794197255459923}},
      {{0, 0, 0}, {0, 0, 0}, {-0.00029927059211173082, 0.00026118075869641392, 0.00035132161602936465},
       {0, 0, 0}},
      {0.93163480449927949, 0.36924891566208573, 0.28743947818824322, -0.78753450712075257},
      {{-0.22862203235631162, 0.05894589575145668, 0.11511810767374644, -0.65256280448438919},
       {-0.4568503872610965, -1.33495587783708, -1.2568222182711835, -0.57268009514914131},
       {1.7422392085597567, -0.56418157997698914, 0.21377690233090399, -0.89421883752649656},
       {-0.058263528637499638, 1.452970897956954, -1.2989615540193649, -0.98318531139972232}},
      {}, 0, 0, {1.0, 1e-4, 0.0, 4, 2}};
  element_geometry<double, double>(q.X, q.c, q.inv, q.rh);
  Results x, ref;
  g_violations = 0;
  by_double<0>(q, ref);
  say("wall_cell_left", 0, 0, by_fixed<0>(q, x) ? 0 : 1, 0);
  say("wall_cell_expect", 0, 0, (double)g_violations, 0);
  Sum s;
  s.add(x, ref);
  say("wall_cell", 0, 0, s.worst(), 1e-12);
}

// Flat cells: component i of the velocity of size scale^i; scale 0: normal
// deviates, some Gauss points of which are nearly at rest. In place, against the
// element in long double, where the double-precision routine's own error (10 %
// for the spread of a finite sample) is the limit, as in check.cpp; rotated,
// where the rounded geometry is common to both, against that routine: two
// results whose errors are a few 1e-16 each.
static Element flat_cell(double flat, double scale, bool rotated) {
  Element q = make(0, 0);
  double R[3][3];
  const double a = rotated ? uni(0, 6.3) : 0, b = rotated ? uni(0, 6.3) : 0;
  const double A[3][3] = {{std::cos(a), -std::sin(a), 0}, {std::sin(a), std::cos(a), 0}, {0, 0, 1}};
  const double B[3][3] = {{std::cos(b), 0, std::sin(b)}, {0, 1, 0}, {-std::sin(b), 0, std::cos(b)}};
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) R[i][j] = A[i][0] * B[0][j] + A[i][1] * B[1][j] + A[i][2] * B[2][j];
  for (int n = 0; n < 4; ++n) {
    const double x[3] = {q.X[n][0], q.X[n][1], q.X[n][2] / flat};
    for (int i = 0; i < 3; ++i) {
      q.X[n][i] = R[i][0] * x[0] + R[i][1] * x[1] + R[i][2] * x[2];
      q.u[n][i] = scale > 0 ? (1 + uni(-0.9, 0.9)) * std::pow(scale, i) : normal();
    }
  }
  element_geometry<double, double>(q.X, q.c, q.inv, q.rh);
  q.P.mu = 1e-4;  // tau from the velocity rather than from the viscosity
  return q;
}
template <int FLAGS>
static void exact_element(const Element& q, ld rhs[4][4], ld vjp[4][4]) {
  typedef std::complex<ld> cld;
  const ld step = 1e-30L;
  for (int b = -1; b < 4; ++b)
    for (int k = 0; k < (b < 0 ? 1 : 4); ++k) {
      cld u[4][3], p[4], F[4][4];
      for (int a = 0; a < 4; ++a) {
        for (int i = 0; i < 3; ++i) u[a][i] = cld(q.u[a][i], a == b && i == k ? step : 0);
        p[a] = cld(q.p[a], a == b && k == 3 ? step : 0);
      }
      reference<FLAGS, cld>(q.X, u, p, q.P, F);
      if (b >= 0) vjp[b][k] = 0;
      for (int a = 0; a < 4; ++a)
        for (int i = 0; i < 4; ++i) {
          if (b < 0) rhs[a][i] = F[a][i].real();
          else vjp[b][k] += q.w[a][i] * (F[a][i].imag() / step);
        }
    }
}
// Errors of a routine against long double, norm-wise per component.
struct Error {
  double d[8] = {}, n[8] = {};
  void add(const Results& x, const ld rhs[4][4], const ld vjp[4][4]) {
    for (int a = 0; a < 4; ++a)
      for (int k = 0; k < 4; ++k) {
        d[k] += std::pow((double)(x.rhs[a][k] - rhs[a][k]), 2);
        n[k] += std::pow((double)rhs[a][k], 2);
        d[4 + k] += std::pow((double)(x.vjp[a][k] - vjp[a][k]), 2);
        n[4 + k] += std::pow((double)vjp[a][k], 2);
      }
  }
  double of(int k) const { return n[k] > 0 ? std::sqrt(d[k] / n[k]) : 0.0; }
};
template <int FLAGS>
static void flat_cells(int n) {
  for (const double flat : {1.0, 20.0, 100.0, 1e3, 1e4})
    for (const double scale : {1.0, 1e-6, 0.0}) {
      if (scale < 1 && (FLAGS & kSkew)) continue;  // the sweep is in double precision there
      const int id = (int)flat * 10 + (scale == 0 ? 2 : scale < 1);
      Error mine, ref;
      Sum turned;
      for (int it = 0; it < n; ++it) {
        Element q = flat_cell(flat, scale, false);
        Results x, y;
        ld rhs[4][4], vjp[4][4];
        by_double<FLAGS>(q, y);
        if (!by_fixed<FLAGS>(q, x)) say("flat_cell_left", FLAGS, id, 1, 0);
        exact_element<FLAGS>(q, rhs, vjp);
        mine.add(x, rhs, vjp);
        ref.add(y, rhs, vjp);
        if (scale < 1) continue;
        q = flat_cell(flat, scale, true);
        by_double<FLAGS>(q, y);
        if (!by_fixed<FLAGS>(q, x)) say("flat_cell_left", FLAGS, id, 1, 0);
        turned.add(x, y);
      }
      for (int k = 0; k < 8; ++k)
        say(k < 4 ? "flat_cell_rhs" : "flat_cell_vjp", FLAGS, 10 * id + k, mine.of(k), 1.1 * ref.of(k));
      if (scale == 1) say("flat_cell_rotated", FLAGS, id, turned.worst(), 2e-15);
    }
}

// Fields that do not vary along an axis, in cells flat or long along it: 0 nothing
// varies, the velocity in the plane only; 1 with a constant velocity across; 2 with
// one that varies in the plane; 3 the cotangent alone does not vary; 4 a channel,
// the velocity u(z) and the pressure p(x). Where the double-precision sums are
// exact, a sum may lose 6 of the 59 bits that its terms have: 2^-53 for each of
// the at most 32 products of a row. Where the double-precision routine has a larger
// error, 4 times that, for the one element that decides a sum over few.
static Element layered(int kind, int axis, double stretch) {
  Element q;
  const Element any = make(0, 0);
  static const int perm[6][3] = {{0, 1, 2}, {1, 2, 0}, {2, 0, 1}, {0, 2, 1}, {2, 1, 0}, {1, 0, 2}};
  const int t = (int)(rng() % 6);
  int l[4][3] = {};
  for (int s = 0; s < 3; ++s) {
    for (int d = 0; d < 3; ++d) l[s + 1][d] = l[s][d];
    l[s + 1][perm[t][s]] += 1;
  }
  if (t >= 3)
    for (int d = 0; d < 3; ++d) std::swap(l[1][d], l[2][d]);
  double field[8][8], off[8][3], at[3];
  for (auto& r : field)
    for (double& x : r) x = normal();
  for (auto& r : off)
    for (double& x : r) x = 0.12 * uni(-1, 1);
  for (double& x : at) x = std::floor(uni(0, 64));
  const int across = 1 << axis;
  for (int a = 0; a < 4; ++a) {
    const int id = l[a][0] | l[a][1] << 1 | l[a][2] << 2, in = id & ~across;
    for (int d = 0; d < 3; ++d)
      q.X[a][d] = (l[a][d] + at[d] + (d == axis ? 0.0 : off[in][d])) / 64 * (d == axis ? stretch : 1);
    for (int k = 0; k < 8; ++k) {
      const bool varies = k > 3 ? kind == 4 : kind == 3;
      double x = field[k][varies ? id : in];
      if (kind == 4 && k < 4) x = field[k][id & (k == 0 ? across : 1 << (axis + 1) % 3)];
      if (k == axis && kind < 2) x = kind;
      if (kind == 4 && k < 3) x = k == 0 ? 0.5 + std::fabs(x) : 0.0;
      if (k < 3) q.u[a][k] = x;
      else if (k == 3) q.p[a] = x;
      else q.w[a][k - 4] = x;
    }
  }
  element_geometry<double, double>(q.X, q.c, q.inv, q.rh);
  q.P = any.P;
  q.P.mu = rng() & 1 ? 1e-2 : 1e-4;
  return q;
}
template <int FLAGS>
static void layers(int n) {
  for (int kind = 0; kind < 5; ++kind)
    for (int axis = 0; axis < 3; ++axis)
      for (const double stretch : {1.0, 0.1, 1e-2, 1e-3, 1e-4, 1e2, 1e4}) {
        Error mine, ref;
        g_violations = 0;
        for (int it = 0; it < n; ++it) {
          const Element q = layered(kind, axis, stretch);
          Results x, y;
          ld rhs[4][4], vjp[4][4];
          by_double<FLAGS>(q, y);
          if (!by_fixed<FLAGS>(q, x)) x = y;  // as the kernels do
          exact_element<FLAGS>(q, rhs, vjp);
          mine.add(x, rhs, vjp);
          ref.add(y, rhs, vjp);
        }
        const int id = (kind * 3 + axis) * 100 + (int)std::lround(10 * std::log10(stretch));
        for (int k = 0; k < 8; ++k)
          say(k < 4 ? "layered_rhs" : "layered_vjp", FLAGS, id * 10 + k, mine.of(k),
              std::max(32 * 0x1p-53, 4 * ref.of(k)));
        say("layered_expect", FLAGS, id, (double)g_violations, 0);
      }
}

template <int FLAGS>
static void all(int n) {
  expectations<FLAGS>(n / 10);
  low_velocities<FLAGS>(n);
}

int main() {
  wall_cell();
  flat_cells<0>(2000);
  flat_cells<kSkew>(1000);
  flat_cells<kTauElem>(1000);
  flat_cells<kSkew | kTauElem>(1000);
  layers<0>(60);
  layers<kSkew>(30);
  layers<kTauElem>(30);
  layers<kSkew | kTauElem>(30);
  all<0>(100000);
  all<1>(20000);
  all<2>(20000);
  all<3>(20000);
  all<4>(20000);
  all<5>(20000);
  all<6>(20000);
  all<7>(20000);
  return 0;
}
