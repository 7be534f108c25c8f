// Host check of the fixed-point node update (csrc/fixed.cuh) against the same collision in long
// double and, for scale, in double. Reads "q r w_0 ... w_(q-1)" from standard input and the state
// ranges from the command line; prints nodes taken, nodes tried, and the root mean square errors
// of populations / (w rho), rho, u_x, T: double first, then fixed point.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#define __host__
#define __device__
#include "../paper_2504_20169_gb300/csrc/fixed.cuh"

using namespace lbm;
typedef long double ld;
static ld W[37], R;

template <class S, class T>
static void equilibrium(T rho, T ux, T uy, T Te, T (&f)[37]) {
  for (int i = 0; i < S::Q; ++i) {
    const T r = (T)R, s = r * (S::ex(i) * ux + S::ey(i) * uy), u2 = ux * ux + uy * uy, th = Te - 1;
    const T c2 = r * r * (S::ex(i) * S::ex(i) + S::ey(i) * S::ey(i));
    T p = 1 + s + (s * s - u2 + th * (c2 - 2)) / 2;
    if (S::ORDER >= 3) p += s / 6 * (s * s - 3 * u2 + 3 * th * (c2 - 4));
    if (S::ORDER >= 4)
      p += (s * s * s * s - 6 * s * s * u2 + 3 * u2 * u2 + 6 * th * (s * s * (c2 - 6) + u2 * (4 - c2)) +
            3 * th * th * (c2 * c2 - 8 * c2 + 8)) / 24;
    f[i] = (T)W[i] * rho * p;
  }
}
template <class S, class T>
static void macro(const T* f, T (&m)[4]) {
  T s = 0, x = 0, y = 0, e = 0;
  for (int i = 0; i < S::Q; ++i) {
    s += f[i];
    x += S::ex(i) * f[i];
    y += S::ey(i) * f[i];
    e += (S::ex(i) * S::ex(i) + S::ey(i) * S::ey(i)) * f[i];
  }
  const T r = (T)R;
  m[0] = s;
  m[1] = r * x / s;
  m[2] = r * y / s;
  m[3] = (r * r * e / s - m[1] * m[1] - m[2] * m[2]) / 2;
}
template <class S, class T>
static void collide(T* f, T omega) {
  T m[4], q[37];
  macro<S, T>(f, m);
  equilibrium<S, T>(m[0], m[1], m[2], m[3], q);
  for (int i = 0; i < S::Q; ++i) f[i] += omega * (q[i] - f[i]);
}
template <class S>
static bool collide_fixed(double* p, const fx::Consts& c) {
  double f[37];
  std::memcpy(f, p, sizeof f);
  int low = 1 << 20, out = 1;
  const fx::Moments m = fx::gather<S>(c, f, 1, low);
  fx::State u;
  if (low < 3 || !fx::state(m, c, u)) return false;
  const fx::Site k = fx::site<S::ORDER>(u, c);
  fx::each_equilibrium<S>(c, k, u.rho, [](const fx::ShellInfo&, int) {},
                          [&](int h, const fx::ShellInfo& s, fx::i64 feq) {
    const fx::i64 F = (fx::i64)fx::bits_of(f[s.first + h]);
    p[s.first + h] = fx::store(fx::relax(F, feq, c.om), s.fe, c.E, out);
  });
  return out >= 1;
}
template <class S>
static void run(double umax, double tmax, double rlo, double rhi, double noise, double omega) {
  fx::Consts c;
  std::memset(&c, 0, sizeof c);
  c.E = (int)std::lround(std::log2(0.5 * (rlo + rhi)));
  c.r2 = fx::split((fx::i64)std::llrint(std::ldexp(R * R, 60)));
  c.inv_r2 = fx::split((fx::i64)std::llrint(std::ldexp(1 / (R * R), 60)));
  c.om = fx::factor((fx::i64)std::llrint(std::ldexp((ld)omega, 61)));
  double w[37];
  for (int i = 0; i < S::Q; ++i) w[i] = (double)W[i];
  if (!fx::make_shells<S>(w, c.shell)) std::exit(3);
  std::mt19937_64 gen(7);
  auto U = [&]() { return std::ldexp((double)(gen() >> 11), -52) - 1.0; };
  const int N = 20000;
  int taken = 0;
  ld e[2][4] = {{0}};
  for (int t = 0; t < N; ++t) {
    const ld a = 3.14159265358979L * U(), v = umax * std::sqrt(std::fabs(U()));
    ld x[37], m0[4], m1[4];
    equilibrium<S, ld>(0.5 * (rlo + rhi) + 0.5 * (rhi - rlo) * U(), v * cosl(a), v * sinl(a),
                       1 + tmax * U(), x);
    double d[37], g[37];
    for (int i = 0; i < S::Q; ++i) x[i] = d[i] = g[i] = (double)(x[i] * (1 + noise * U()));
    if (!collide_fixed<S>(g, c)) continue;
    ++taken;
    collide<S, ld>(x, omega);
    collide<S, double>(d, omega);
    macro<S, ld>(x, m0);
    for (int k = 0; k < 2; ++k) {
      ld y[37], p = 0;
      for (int i = 0; i < S::Q; ++i) {
        y[i] = k ? g[i] : d[i];
        p += (y[i] - x[i]) * (y[i] - x[i]) / (W[i] * m0[0] * W[i] * m0[0]);
      }
      macro<S, ld>(y, m1);
      e[k][0] += p / S::Q;
      e[k][1] += (m1[0] - m0[0]) * (m1[0] - m0[0]);
      e[k][2] += (m1[1] - m0[1]) * (m1[1] - m0[1]);
      e[k][3] += (m1[3] - m0[3]) * (m1[3] - m0[3]);
    }
  }
  std::printf("%d %d", taken, N);
  for (int k = 0; k < 2; ++k)
    for (int j = 0; j < 4; ++j) std::printf(" %.6Le", taken ? sqrtl(e[k][j] / taken) : 0.0L);
  std::printf("\n");
}
int main(int argc, char** argv) {
  int q;
  if (argc != 7 || std::scanf("%d %Lf", &q, &R) != 2) return 2;
  for (int i = 0; i < q; ++i)
    if (std::scanf("%Lf", &W[i]) != 1) return 2;
  double a[6];
  for (int k = 0; k < 6; ++k) a[k] = std::atof(argv[k + 1]);
  if (q == 37) run<D2Q37>(a[0], a[1], a[2], a[3], a[4], a[5]);
  else if (q == 17) run<D2Q17>(a[0], a[1], a[2], a[3], a[4], a[5]);
  else run<D2Q9>(a[0], a[1], a[2], a[3], a[4], a[5]);
  return 0;
}
