// Host check of the limits of fixed.cuh's range. Reads "q r w_0 ... w_(q-1)" from standard input.
// First line: of states on either side of a limit, those taken and those refused (inside taken,
// inside tried, outside taken, outside tried). Second line, over states on the limits themselves and
// in their corners: the largest |f_eq| and the largest difference from long double, both in
// population units.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#define __host__
#define __device__
#include "../paper_2504_20169_gb300/csrc/fixed.cuh"

using namespace lbm;
typedef long double ld;
static double W[37], R;

static fx::i64 units(ld v, int e) { return (fx::i64)llrintl(ldexpl(v, e)); }
static fx::Moments moments_of(ld rho, ld X, ld Y, ld T) {   // X, Y = r u
  const ld r2 = (ld)R * R;
  return {units(rho, 58), units(rho * X / r2, 58), units(rho * Y / r2, 58),
          units(rho * (2 * T + (X * X + Y * Y) / r2) / r2, 58)};
}

template <class S>
static int run() {
  fx::Consts c;
  std::memset(&c, 0, sizeof c);
  c.r2 = fx::split(units((ld)R * R, 60));
  c.inv_r2 = fx::split(units(1 / ((ld)R * R), 60));
  if (!fx::make_shells<S>(W, c.shell)) return 3;
  std::mt19937_64 gen(3);
  auto U = [&]() { return std::ldexp((double)(gen() >> 11), -52) - 1.0; };
  const ld rest[4] = {1, 0, 0, 1}, eps = 1e-9L;
  int n[4] = {0, 0, 0, 0};
  for (int t = 0; t < 6000; ++t) {
    // one quantity at its limit, the others anywhere inside (every eighth time at rest)
    const ld a = 3.14159265358979323846L * U(), m = t % 8 ? 1.0L : 0.0L;
    ld rho = m ? exp2l(0.99L * U()) : rest[0], v = m * sqrtl(0.6L * fabsl(U())), T = 1 + m * 0.24L * U();
    const int side = t % 2;
    const ld d = side ? eps : -eps;   // outwards, inwards
    switch (t / 2 % 5) {
      case 0: rho = 2 * (1 + d); break;
      case 1: rho = 0.5L * (1 - d); break;
      case 2: v = sqrtl(0.7L) * (1 + d); break;
      case 3: T = 1.25L + d; break;
      case 4: T = 0.75L - d; break;
    }
    fx::State u, u2;
    const bool in = fx::state(moments_of(rho, v * cosl(a), v * sinl(a), T), c, u);
    const bool in2 = fx::state_of((double)rho, (double)(v * cosl(a)), (double)(v * sinl(a)),
                                  (double)T, c, u2);
    if (in != in2) return 4;
    n[2 * side] += in;
    n[2 * side + 1] += 1;
  }
  std::printf("%d %d %d %d\n", n[0], n[1], n[2], n[3]);
  ld most = 0, worst = 0;
  for (int t = 0; t < 40000; ++t) {
    fx::State u;
    const ld a = t < 16 ? 3.14159265358979323846L / 8 * t : 3.14159265358979323846L * U();
    const ld X = sqrtl(0.7L) * cosl(a), Y = sqrtl(0.7L) * sinl(a), th = t % 2 ? 0.25L : -0.25L;
    u.rho = (1ll << 59) - 1;
    u.X = units(X, 60);
    u.Y = units(Y, 60);
    u.th = units(t % 4 < 2 ? th : th * U(), 60);
    const ld rho = ldexpl(u.rho, -58), x = ldexpl(u.X, -60), y = ldexpl(u.Y, -60), h = ldexpl(u.th, -60);
    const ld r2 = (ld)R * R, v2 = (x * x + y * y) / r2;
    const fx::Site k = fx::site<S::ORDER>(u, c);
    fx::each_equilibrium<S>(c, k, u.rho, [](const fx::ShellInfo&, int) {},
                            [&](int j, const fx::ShellInfo& s, fx::i64 feq) {
      const int i = s.first + j;
      const ld q = S::ex(i) * x + S::ey(i) * y, c2 = r2 * (S::ex(i) * S::ex(i) + S::ey(i) * S::ey(i));
      ld p = 1 + q + (q * q - v2 + h * (c2 - 2)) / 2;
      if (S::ORDER >= 3) p += q / 6 * (q * q - 3 * v2 + 3 * h * (c2 - 4));
      if (S::ORDER >= 4)
        p += (q * q * q * q - 6 * q * q * v2 + 3 * v2 * v2 + 6 * h * (q * q * (c2 - 6) + v2 * (4 - c2)) +
              3 * h * h * (c2 * c2 - 8 * c2 + 8)) / 24;
      const ld f = ldexpl((ld)W[i] * rho * p, s.fe);
      most = std::max(most, fabsl(f));
      worst = std::max(worst, fabsl((ld)feq - f));
    });
  }
  std::printf("%.6Le %.3Lf\n", most, worst);
  return 0;
}

int main() {
  int q;
  if (std::scanf("%d %lf", &q, &R) != 2) return 2;
  for (int i = 0; i < q; ++i)
    if (std::scanf("%lf", &W[i]) != 1) return 2;
  return q == 37 ? run<D2Q37>() : q == 17 ? run<D2Q17>() : run<D2Q9>();
}
