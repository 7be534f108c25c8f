// The FP64 node update in 64-bit fixed point.
//
// GB300 issues one FP64 instruction per warp in 64 cycles and quadrant of an SM (76 when all four
// quadrants do), measured; a 64-bit integer add takes 3 cycles and a 64 x 62 bit product about 20.
// A D2Q37 update has about 390 FP64 instructions, most of them additions, so the FP64 kernels are
// bound by that pipe at a tenth of the memory bandwidth. Here populations are exact integers from
// load to store, and FP64 is left with the site's scalars (about 70 operations per node).
//
// Formats. A population of a shell with weight w is F = f 2^(fe - E), fe = 57 + k with
// w 2^k in (1/2, 1) (two bits less on the outer shells n = |e|^2 >= 8, whose equilibrium factor
// spans four times the range), E = the exponent of the mean density: near the state of rest one
// unit of F is 2^-56 of the population (2^-54 on the outer shells), an eighth of the unit in the
// last place of its double. Reading a double is exact down to a small fraction of the rest
// population; products are rounded to nearest with the mean of their dropped low part added (no
// bias), and the store rounds to nearest. So each population is off by less than in FP64, whose
// equilibrium rounds several times at 2^-53.
// The equilibrium factor P = f_eq / (w rho) is an integer polynomial in the lattice velocity with
// the site's scalars, in units of 2^-60 (2^-58 on the outer shells).
//
// Range. A node takes this path if every population is in [0, 2^59) units, 1/2 < rho 2^-E < 2,
// |r u|^2 <= 0.7 (|u| <= 0.7 on D2Q37) and |T - 1| <= 1/4: then |P| < 8 (32 on the outer shells)
// and no sum or product leaves its integer. Every other node (NaN and infinities too) takes the
// FP64 arithmetic.
//
// Host and device: everything here compiles for both, so the arithmetic can be checked on a CPU.
#pragma once
#include <cstdint>
#include <cstring>
#include <utility>

#include "stencils.cuh"

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#include <cmath>
#endif

namespace lbm {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

// fn(integral_constant<0>) ... fn(integral_constant<N - 1>): arrays indexed inside stay in registers
template <class Fn, int... I>
LBM_HD void unroll_seq(Fn&& fn, std::integer_sequence<int, I...>) {
  (fn(std::integral_constant<int, I>()), ...);
}
template <int N, class Fn>
LBM_HD void unroll(Fn&& fn) {
  unroll_seq(fn, std::make_integer_sequence<int, N>());
}

LBM_HD u64 bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(v);
#else
  u64 b;
  std::memcpy(&b, &v, 8);
  return b;
#endif
}
LBM_HD double double_of(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)b);
#else
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
LBM_HD int clz(u64 v) {
#ifdef __CUDA_ARCH__
  return __clzll((i64)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
LBM_HD int clz32(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
// v >> s for s >= 0, zero from 64 on
LBM_HD u64 shr(u64 v, int s) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}
LBM_HD u64 shl(u64 v, int s) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s > 63 ? 0 : v << s;
#endif
}

// A factor 0 <= v < 2^62 as two 32-bit limbs, v = h 2^32 + l with l signed, so that every
// partial product with a 64-bit integer is one native 32 x 32 -> 64 bit multiplication.
struct Limbs {
  unsigned h;
  int l;
};
LBM_HD Limbs split(i64 v) {
  const u64 r = (u64)v + 0x80000000u;
  return Limbs{(unsigned)(r >> 32), (int)(unsigned)v};
}

// a b / 2^64, off by less than one unit and by none on average: the product of the low limbs
// (mean 0, as l is signed) is left out, and 2^31 rounds.
LBM_HD i64 mul(i64 a, Limbs b) {
  const int ah = (int)(a >> 32);
  i64 m = (i64)ah * b.l + (1ll << 31);
  m += (i64)((u64)(unsigned)a * b.h);
  return (i64)ah * (int)b.h + (m >> 32);
}

// Weight exponent of a shell: w 2^k in (1/2, 1) (checked when a context is created).
template <class S>
LBM_HD constexpr int shell_k(int s) {
  if (S::Q == 37) {
    constexpr int t[8] = {2, 3, 4, 6, 7, 9, 11, 11};
    return t[s];
  }
  if (S::Q == 17) {
    constexpr int t[8] = {1, 3, 4, 13, 11, 0, 0, 0};
    return t[s];
  }
  constexpr int t[8] = {1, 3, 5, 0, 0, 0, 0, 0};
  return t[s];
}
template <class S>
LBM_HD constexpr int shell_n(int s) {
  return S::shell_a(s) * S::shell_a(s) + S::shell_b(s) * S::shell_b(s);
}
// bits by which an outer shell is coarser
template <class S>
LBM_HD constexpr int shell_far(int s) {
  return shell_n<S>(s) >= 8 ? 2 : 0;
}
template <class S>
LBM_HD constexpr int shell_fe(int s) {
  return 57 + shell_k<S>(s) - shell_far<S>(s);
}

// f 2^(fe - E) of a double f >= 0. `low` takes the smallest right shift seen: below 3 a
// population is out of range (2^59 units or more, negative, infinite or NaN).
LBM_HD i64 load(double f, int fe, int E, int& low) {
  const u64 b = bits_of(f);
  const unsigned hi = (unsigned)(b >> 32);
  const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u)) << 32 | (unsigned)b) << 9;   // top bit 61
  const int s = 1084 - fe + E - (int)(hi >> 20);   // the sign bit makes this negative
  low = s < low ? s : low;
  return (i64)shr(m, s < 0 ? 0 : s);
}

// The double nearest to F 2^(E - fe) for 2^32 <= F < 2^62; `low` takes the smallest upper word
// seen: below 1 a value is out of this range (a population that is negative or 2^-25 of its
// weight) and the result is not the value.
LBM_HD double store(i64 F, int fe, int E, int& low) {
  const int fh = (int)(F >> 32);
  low = fh < low ? fh : low;
  const int z = clz32((unsigned)fh);
  const u64 r = (shl((u64)F, z - 1) + 0x200) >> 10;   // 53 bits, rounded; a carry moves the exponent up
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(1023 + 62 - fe + E - z) << 20);
  return double_of((u64)hi << 32 | (unsigned)r);
}
// Any |F| < 2^62, zero and negative included.
LBM_HD double store(i64 F, int fe, int E) {
  const i64 sg = F >> 63;
  const u64 m = (u64)((F ^ sg) - sg);
  const int z = clz(m);
  const u64 r = (shl(m, z - 1) + 0x200) >> 10;
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(1023 + 62 - fe + E - z) << 20) +
                      ((unsigned)(F >> 32) & 0x80000000u);
  return m ? double_of((u64)hi << 32 | (unsigned)r) : 0.0;
}

// A site scalar |v| < 8 in units of 2^-60, truncated.
LBM_HD i64 scalar(double v) {
  const u64 b = bits_of(v);
  const unsigned hi = (unsigned)(b >> 32);
  const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u)) << 32 | (unsigned)b) << 10;   // top bit 62
  const i64 a = (i64)shr(m, 1025 - (int)((hi >> 20) & 0x7ff));
  const i64 sg = (i64)b >> 63;
  return (a ^ sg) - sg;
}

// Constants of a context: the shells' weights w 2^k in units of 2^-62, the relaxation rate in
// units of 2^-61, the exponent E, and the mean equilibrium in each direction's units.
struct Consts {
  Limbs w[8], om;
  double r2, inv_r2;
  int E;
  int on;          // 0: FP64 arithmetic everywhere (omega = 0 keeps populations bit for bit)
  i64 eqbar[37];
};

// Scalars of the equilibrium polynomial: with integer velocity (a, b), n = a^2 + b^2,
//   even part  A0 + n A1 + n^2 A2 + a^2 b^2 B + (a^2 - b^2)(P0 + n P1)
//              + a b (Q0 + n Q1 + (a^2 - b^2) Q2)
//   odd part   a (Rx0 + n Rx1 + a^2 Tx) + b (Ry0 + n Ry1 + b^2 Ty),
// Eqs. (feq-2/3/4) with xi = r e sorted by their behaviour under the symmetries of the square.
struct Site {
  i64 A0, A1, A2, B, P0, P1, Q0, Q1, Q2, Rx0, Rx1, Tx, Ry0, Ry1, Ty;
};

// X = r u_x, Y = r u_y, theta = T - 1. |X|^2 + |Y|^2 <= 0.7 and |theta| <= 1/4 keep every
// scalar below 4.
template <int ORDER>
LBM_HD Site site(double X, double Y, double th, double r2, double inv_r2) {
  const double p = X * X, m = Y * Y, xy = X * Y, S = p + m, D = p - m;
  const double u2 = S * inv_r2, rt = r2 * th;
  Site k;
  k.A2 = k.B = k.P1 = k.Q1 = k.Q2 = k.Rx1 = k.Tx = k.Ry1 = k.Ty = 0;
  const double one = 1.0 - 0.5 * u2;
  if (ORDER >= 4) {
    const double half = 0.5 - 0.25 * u2;
    const double k20 = half - 1.5 * th;
    const double x4 = S * S - 2.0 * (p * m);
    const double z = S * (1.0 / 48.0) + 0.125 * rt;
    k.A0 = scalar((one - th) + th * (th + u2) + 0.125 * (u2 * u2));
    k.A1 = scalar(rt * (half - th) + 0.5 * (k20 * S));
    k.A2 = scalar(0.125 * (rt * (rt + S)) + x4 * (1.0 / 48.0));
    k.B = scalar(0.25 * (p * m) - x4 * (1.0 / 24.0));
    k.P0 = scalar(0.5 * (k20 * D));
    k.P1 = scalar(z * D);
    k.Q0 = scalar(2.0 * (xy * k20));
    k.Q1 = scalar(4.0 * (xy * z));
    k.Q2 = scalar(xy * (D * (1.0 / 12.0)));
  } else {
    k.A0 = scalar(one - th);
    k.A1 = scalar(0.5 * rt + 0.25 * S);
    k.P0 = scalar(0.25 * D);
    k.Q0 = scalar(xy);
  }
  if (ORDER >= 3) {
    const double k10 = one - 2.0 * th;
    k.Rx0 = scalar(X * k10);
    k.Ry0 = scalar(Y * k10);
    k.Rx1 = scalar(0.5 * (X * (rt + m)));
    k.Ry1 = scalar(0.5 * (Y * (rt + p)));
    k.Tx = scalar((X * (1.0 / 6.0)) * (p - 3.0 * m));
    k.Ty = scalar((Y * (1.0 / 6.0)) * (m - 3.0 * p));
  } else {
    k.Rx0 = scalar(X);
    k.Ry0 = scalar(Y);
  }
  return k;
}

// The scalars in the outer shells' units.
template <int ORDER>
LBM_HD Site coarse(const Site& k) {
  Site c;
  c.A0 = k.A0 >> 2; c.A1 = k.A1 >> 2; c.P0 = k.P0 >> 2; c.Q0 = k.Q0 >> 2;
  c.Rx0 = k.Rx0 >> 2; c.Ry0 = k.Ry0 >> 2;
  c.A2 = c.B = c.P1 = c.Q1 = c.Q2 = c.Rx1 = c.Tx = c.Ry1 = c.Ty = 0;
  if (ORDER >= 4) {
    c.A2 = k.A2 >> 2; c.B = k.B >> 2; c.P1 = k.P1 >> 2; c.Q1 = k.Q1 >> 2; c.Q2 = k.Q2 >> 2;
  }
  if (ORDER >= 3) {
    c.Rx1 = k.Rx1 >> 2; c.Tx = k.Tx >> 2; c.Ry1 = k.Ry1 >> 2; c.Ty = k.Ty >> 2;
  }
  return c;
}

// What the directions of a shell (a, b) share; a direction with |e_x| = a is of kind 0, with
// |e_x| = b of kind 1 (the axes swapped).
struct Shell {
  i64 even[2];       // symmetric in both components
  i64 cross[2];      // times the sign of e_x e_y
  i64 x[2], y[2];    // times the sign of e_x, of e_y
};
template <class S>
LBM_HD Shell shell(const Site& k, int s) {
  const int a = S::shell_a(s), b = S::shell_b(s), n = a * a + b * b, d = a * a - b * b;
  Shell h;
  i64 sym = k.A0 + n * k.A1, anti = k.P0, q = k.Q0, ux = k.Rx0, uy = k.Ry0;
  if (S::ORDER >= 4) {
    sym += (n * n) * k.A2 + (a * a * b * b) * k.B;
    anti += n * k.P1;
    q += n * k.Q1;
  }
  if (S::ORDER >= 3) {
    ux += n * k.Rx1;
    uy += n * k.Ry1;
  }
  h.even[0] = sym + d * anti;
  h.even[1] = sym - d * anti;
  const i64 q0 = (a * b) * q, q2 = S::ORDER >= 4 ? (a * b * d) * k.Q2 : 0;
  h.cross[0] = q0 + q2;
  h.cross[1] = q0 - q2;
  h.x[0] = a * ux;
  h.x[1] = b * ux;
  h.y[0] = b * uy;
  h.y[1] = a * uy;
  if (S::ORDER >= 3) {
    h.x[0] += (a * a * a) * k.Tx;
    h.x[1] += (b * b * b) * k.Tx;
    h.y[0] += (b * b * b) * k.Ty;
    h.y[1] += (a * a * a) * k.Ty;
  }
  return h;
}
// Even and odd part of P of one direction of the shell.
template <class S>
LBM_HD void factor(const Shell& h, int s, int ex, int ey, i64& even, i64& odd) {
  const int kind = (ex < 0 ? -ex : ex) == S::shell_a(s) ? 0 : 1;
  even = h.even[kind];
  if (ex * ey > 0) even += h.cross[kind];
  if (ex * ey < 0) even -= h.cross[kind];
  odd = ex > 0 ? h.x[kind] : ex < 0 ? -h.x[kind] : 0;
  if (ey > 0) odd += h.y[kind];
  if (ey < 0) odd -= h.y[kind];
}

// The weight of a shell times the density (rho 2^-E in units of 2^-58), in units of 2^-61: the
// second factor of every direction's equilibrium, below 2^62.
template <class S>
LBM_HD Limbs shell_weight(const Consts& c, int s, i64 rho58) {
  return split(2 * mul(rho58 << 4, c.w[s]));
}

// f_eq in the direction's units from P (units of 2^-60, on the outer shells 2^-58).
LBM_HD i64 equilibrium(i64 P, Limbs wr) { return mul(P, wr); }

// F + omega (feq - F); |feq - F| < 2^60.
LBM_HD i64 relax(i64 F, i64 feq, Limbs om) { return F + mul((feq - F) * 8, om); }

// Moments of a node's populations: rho, sum f e_x, sum f e_y, sum f |e|^2 (times 2^-E), in
// units of 2^-58. Each shell is summed exactly (at most eight values below 2^59) and then
// rounded to the common unit.
struct Moments {
  i64 rho, jx, jy, e2;
};
template <class S>
LBM_HD Moments moments(const i64 (&F)[S::Q]) {
  Moments m{0, 0, 0, 0};
  unroll<S::NSHELL>([&](auto sc) {
    constexpr int s = sc, i0 = S::shell_first(s), size = S::shell_size(s);
    constexpr int sh = shell_fe<S>(s) - 58;
    constexpr i64 half = (1ll << sh) >> 1;
    if constexpr (size == 1) {
      m.rho += (F[i0] + half) >> sh;
    } else {
      i64 sum = half, x = half, y = half;
      unroll<size / 2>([&](auto h) {
        constexpr int ip = i0 + h, im = ip + size / 2;
        const i64 a = F[ip], b = F[im];
        sum += a + b;
        x += S::ex(ip) * (a - b);
        y += S::ey(ip) * (a - b);
      });
      sum >>= sh;
      m.rho += sum;
      m.jx += x >> sh;
      m.jy += y >> sh;
      m.e2 += shell_n<S>(s) * sum;
    }
  });
  return m;
}

// 1 / v for v in (2^57, 2^59): Newton's iteration from the single-precision reciprocal of the
// leading bits (conversions to and from FP64 run in the FP64 pipe: the seed avoids them).
LBM_HD double reciprocal(i64 v) {
  const float f = 1.0f / (float)(int)(v >> 28);
  unsigned fb;
#ifdef __CUDA_ARCH__
  fb = __float_as_uint(f);
#else
  std::memcpy(&fb, &f, 4);
#endif
  const double x0 = double_of(((u64)fb << 29) + ((u64)(1023 - 127 - 28) << 52)), d = (double)v;
  const double x1 = fma(x0, fma(-d, x0, 1.0), x0);
  return fma(x1, fma(-d, x1, 1.0), x1);
}

// Macroscopic state of a node in range.
struct State {
  i64 rho;            // units of 2^-58, times 2^-E
  double X, Y, th;    // r u and T - 1
};

LBM_HD bool state(const Moments& m, const Consts& c, State& u) {
  if (m.rho <= (1ll << 57) || m.rho >= (1ll << 59)) return false;
  const double inv = reciprocal(m.rho), ri = c.r2 * inv;
  u.rho = m.rho;
  u.X = (double)m.jx * ri;
  u.Y = (double)m.jy * ri;
  // D rho T = r^2 sum f |e|^2 - rho u^2 with D = 2 and u = (X, Y) / r
  const double s = u.X * u.X + u.Y * u.Y;
  u.th = 0.5 * ((double)m.e2 * ri - s * c.inv_r2) - 1.0;
  return s <= 0.7 && u.th <= 0.25 && u.th >= -0.25;
}

}  // namespace fx
}  // namespace lbm
