// The FP64 node update in 64-bit fixed point.
//
// GB300 issues one FP64 instruction per warp in 64 cycles and quadrant of an SM (76 when all four
// quadrants do), measured; a 64-bit integer add takes 3 cycles and a 64 x 62 bit product about 20.
// A D2Q37 update has about 390 FP64 instructions, most of them additions, so the FP64 kernels are
// bound by that pipe at a tenth of the memory bandwidth. Here a node is integers from load to
// store: populations, moments, the scalars of its equilibrium and the relaxation.
//
// Formats. A population of a shell with weight w is F = f 2^(fe - E), fe = 55 + k with
// w 2^k in (1/2, 1), E = the exponent of the mean density: near the state of rest one unit of F is
// 2^-54 to 2^-55 of the population, a half to a quarter of the unit in the last place of its
// double. Reading a double down to about a quarter of its weight is exact; a smaller one is rounded
// down to a unit, which drops bits only of what FP64 arithmetic wrote (an initial state, PML terms,
// a neighbour out of range): what this update stores are whole units. Products are rounded to
// nearest with the mean of their dropped low part added (no bias), and the store rounds to nearest.
// So each population is off by less than in FP64, whose equilibrium rounds several times at 2^-53 of its
// terms, small population or not. (Rounding to nearest in the load too: D2Q37 interior at 1024^2
// 207 -> 216 us, and 800 steps of uniform flows to the same bits.)
// Velocity, temperature and what follows from them are in units of 2^-60 (FP64 has 2^-53 of the
// value). The equilibrium factor P = f_eq / (w rho) is an integer polynomial in the lattice
// velocity with the site's scalars, in units of 2^-58.
//
// Range. A node takes this path if every population is in [0, 2^59) units, 1/2 < rho 2^-E < 2,
// |r u|^2 <= 0.7 (|u| <= 0.7 on D2Q37) and |T - 1| <= 1/4: then |P| < 32 and no sum or product
// leaves its integer. Every other node (NaN and infinities too) takes the FP64 arithmetic.
//
// Layout. A thread keeps its node in shared memory (value i at f[i * stride]) and walks the shells
// in rolled loops, one for each of the three kinds of shell: unrolled over the directions with
// everything in registers the code is 70 KB and misses the instruction cache, and 128 registers
// a thread leave four warps to a scheduler.
//
// Host and device: everything here compiles for both, so the arithmetic can be checked on a CPU.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "stencils.cuh"

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

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
// 2^e, -1022 <= e <= 1023
LBM_HD double pow2(int e) { return double_of((u64)(unsigned)(1023 + e) << 52); }
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

// A factor |v| < 2^63 as two signed 32-bit limbs, v = h 2^32 + l: every partial product is one
// native 32 x 32 -> 64 bit multiplication.
struct Limbs {
  int h, l;
};
LBM_HD Limbs split(i64 v) {
  const u64 r = (u64)v + 0x80000000u;
  return Limbs{(int)(r >> 32), (int)(unsigned)v};
}

// A factor 0 <= v < 2^62 of many products: its limbs and the constant that rounds them.
struct Factor {
  int h, l;
  unsigned c;        // 2^31 + l / 2
};
LBM_HD Factor factor(i64 v) {
  const Limbs b = split(v);
  return Factor{b.h, b.l, 0x80000000u + (unsigned)(b.l >> 1)};
}

// a b / 2^64, off by less than one unit and by none on average: the product of the low limbs is
// replaced by its mean over the low limb of a, and 2^31 rounds.
LBM_HD i64 mul(i64 a, Factor b) {
  const int ah = (int)(a >> 32);
  i64 m = (i64)ah * b.l + (i64)(u64)b.c;
  m += (i64)((u64)(unsigned)a * (unsigned)b.h);
  return (i64)ah * b.h + (m >> 32);
}

// a b in units of 2^-TO for a, b in units of 2^-60 (|a| + |b| < 16), off by 2^(TO - 58) at most.
template <int TO = 60>
LBM_HD i64 prod(Limbs a, Limbs b) {
  constexpr int up = TO - 56;
  i64 m = (i64)a.h * b.l + (1ll << (31 - up));
  m += (i64)a.l * b.h;
  return (i64)((u64)((i64)a.h * b.h) << up) + (m >> (32 - up));
}

// Kinds of shell: (0, 0), then (a, 0), then (a, a), then (a, b).
template <class S>
LBM_HD constexpr int kind_of(int s) {
  return S::shell_a(s) == 0 ? 0 : S::shell_b(s) == 0 ? 1 : S::shell_a(s) == S::shell_b(s) ? 2 : 3;
}
template <class S>
LBM_HD constexpr int kind_count(int kind) {
  int n = 0;
  for (int s = 0; s < S::NSHELL; ++s) n += kind_of<S>(s) == kind ? 1 : 0;
  return n;
}

// Position of a direction's shell in the order of kinds.
template <class S>
LBM_HD constexpr int shell_position(int i) {
  int at = 0, mine = 0;
  for (int s = 0; s < S::NSHELL; ++s)
    if (i >= S::shell_first(s)) mine = s;
  for (int s = 0; s < S::NSHELL; ++s)
    if (kind_of<S>(s) < kind_of<S>(mine) || (kind_of<S>(s) == kind_of<S>(mine) && s < mine)) ++at;
  return at;
}
// The shells of one of four warps that share 32 nodes: at most 12 of 37 directions, 5 of 17, 4 of 9.
template <class S>
LBM_HD unsigned warp_shells(int w) {
  if (S::Q == 37) return w == 0 ? 0x40u : w == 1 ? 0x80u : w == 2 ? 0x07u : 0x38u;
  if (S::Q == 17) return w == 0 ? 0x02u : w == 1 ? 0x04u : w == 2 ? 0x08u : 0x11u;
  return w == 0 ? 0x02u : w == 1 ? 0x04u : w == 2 ? 0x01u : 0x00u;
}

// A shell as the loops see it: velocities of base (a, b), a >= b, from direction `first` on.
struct ShellInfo {
  int first, a, b, fe;
  Factor w;          // weight w 2^k in units of 2^-62
};

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

// The leading 53 bits of a value with its top bit at 62, to nearest, halves to even (with two to
// four bits to drop, halves are common); a carry moves the exponent up where it is added.
LBM_HD u64 round53(u64 n) { return (n + 0x1ff + ((unsigned)(n >> 10) & 1u)) >> 10; }

// The double nearest to F 2^(E - fe) for 2^32 <= F < 2^62; `low` takes the smallest upper word
// seen: below 1 a value is out of this range (a population that is negative or 2^-25 of its
// weight) and the result is not the value.
LBM_HD double store(i64 F, int fe, int E, int& low) {
  const int fh = (int)(F >> 32);
  low = fh < low ? fh : low;
  const int z = clz32((unsigned)fh);
  const u64 r = round53(shl((u64)F, z - 1));
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(1023 + 62 - fe + E - z) << 20);
  return double_of((u64)hi << 32 | (unsigned)r);
}
// Any |F| < 2^62, zero and negative included.
LBM_HD double store(i64 F, int fe, int E) {
  const i64 sg = F >> 63;
  const u64 m = (u64)((F ^ sg) - sg);
  const int z = clz(m);
  const u64 r = round53(shl(m, z - 1));
  const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(1023 + 62 - fe + E - z) << 20) +
                      ((unsigned)(F >> 32) & 0x80000000u);
  return m ? double_of((u64)hi << 32 | (unsigned)r) : 0.0;
}

// |v| < 8 in units of 2^-60, truncated.
LBM_HD i64 fixed60(double v) {
  const u64 b = bits_of(v);
  const unsigned hi = (unsigned)(b >> 32);
  const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u)) << 32 | (unsigned)b) << 10;   // top bit 62
  const i64 a = (i64)shr(m, 1025 - (int)((hi >> 20) & 0x7ff));
  const i64 sg = (i64)b >> 63;
  return (a ^ sg) - sg;
}

// Constants of a context: the shells ordered by kind, the relaxation rate in units of 2^-61, the
// exponent E, and the mean equilibrium in each direction's units.
struct Consts {
  ShellInfo shell[8];
  Factor om;
  Limbs r2, inv_r2;  // r^2 and 1 / r^2 in units of 2^-60
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

// Macroscopic state of a node in range.
struct State {
  i64 rho;           // rho 2^-E in units of 2^-58
  i64 X, Y, th;      // r u and T - 1 in units of 2^-60
};

// v / 4, to nearest, halves to even: rounding these scalars down would lose 1e-17 of rho and T in
// every step.
LBM_HD i64 quarter(i64 v) { return (v + 1 + ((unsigned)(v >> 2) & 1u)) >> 2; }

// From the state: |X|^2 + |Y|^2 <= 0.7 and |theta| <= 1/4 keep every value here below 4.
template <int ORDER>
LBM_HD Site site(const State& u, const Consts& c) {
  const i64 ONE = 1ll << 60;
  const Limbs X = split(u.X), Y = split(u.Y), th = split(u.th);
  const i64 p = prod(X, X), m = prod(Y, Y), xy = prod(X, Y), S = p + m, D = p - m;
  const Limbs Ss = split(S), Ds = split(D), xs = split(xy);
  const i64 u2 = prod(Ss, c.inv_r2), rt = prod(c.r2, th);
  const i64 one = ONE - (u2 >> 1);
  // 1/48, 1/12 and 1/6 in units of 2^-60
  const Limbs k48 = split(ONE / 48), k12 = split(ONE / 12), k6 = split(ONE / 6);
  Site k;
  k.A2 = k.B = k.P1 = k.Q1 = k.Q2 = k.Rx1 = k.Tx = k.Ry1 = k.Ty = 0;
  if (ORDER >= 4) {
    const i64 half = (ONE >> 1) - (u2 >> 2);
    const Limbs k20 = split(half - u.th - (u.th >> 1)), rs = split(rt), us = split(u2);
    const i64 pm = prod(xs, xs), x48 = prod(split(prod(Ss, Ss) - 2 * pm), k48);
    const Limbs t = split(S + 6 * rt);
    k.A0 = quarter(one - u.th + prod(th, split(u.th + u2)) + (prod(us, us) >> 3));
    k.A1 = quarter(prod(rs, split(half - u.th)) + (prod(k20, Ss) >> 1));
    k.A2 = quarter((prod(rs, split(rt + S)) >> 3) + x48);
    k.B = quarter((pm >> 2) - 2 * x48);
    const Limbs x12 = split(prod(xs, k12));
    k.P0 = prod<57>(k20, Ds);
    k.P1 = prod<58>(t, split(prod(Ds, k48)));
    k.Q0 = prod<59>(xs, k20);
    k.Q1 = prod<58>(t, x12);
    k.Q2 = prod<58>(Ds, x12);
  } else {
    k.A0 = quarter(one - u.th);
    k.A1 = quarter((rt >> 1) + (S >> 2));
    k.P0 = D >> 4;
    k.Q0 = quarter(xy);
  }
  if (ORDER >= 3) {
    const Limbs k10 = split(one - 2 * u.th);
    k.Rx0 = prod<58>(X, k10);
    k.Ry0 = prod<58>(Y, k10);
    k.Rx1 = prod<57>(X, split(rt + m));
    k.Ry1 = prod<57>(Y, split(rt + p));
    k.Tx = prod<58>(X, split(prod(split(p - 3 * m), k6)));
    k.Ty = prod<58>(Y, split(prod(split(m - 3 * p), k6)));
  } else {
    k.Rx0 = quarter(u.X);
    k.Ry0 = quarter(u.Y);
  }
  return k;
}

// The weight of a shell times the density (rho 2^-E in units of 2^-58), in units of 2^-61: the
// second factor of every direction's equilibrium, below 2^62.
LBM_HD Factor shell_weight(const ShellInfo& h, i64 rho58) { return factor(2 * mul(rho58 << 4, h.w)); }

// F + omega (feq - F); |feq - F| < 2^60.
LBM_HD i64 relax(i64 F, i64 feq, Factor om) { return F + mul((feq - F) * 8, om); }

constexpr unsigned kAllShells = 0xffu;

// put(h, shell, feq) for every direction shell.first + h with its equilibrium in fixed point;
// pre(shell, size) before a shell (h and size are integral constants). Only the shells in `mask`
// (bit k: c.shell[k]).
template <class S, class Pre, class Put>
LBM_HD void each_equilibrium(const Consts& c, const Site& k, i64 rho58, Pre pre, Put put,
                             unsigned mask = kAllShells) {
  constexpr int axis = kind_count<S>(1), diag = kind_count<S>(2), octet = kind_count<S>(3);
  using std::integral_constant;
  integral_constant<int, 0> h0;
  integral_constant<int, 1> h1;
  integral_constant<int, 2> h2;
  integral_constant<int, 3> h3;
  integral_constant<int, 4> h4;
  integral_constant<int, 5> h5;
  integral_constant<int, 6> h6;
  integral_constant<int, 7> h7;
  integral_constant<int, 8> h8;
  if (mask & 1u) {
    const ShellInfo& h = c.shell[0];
    pre(h, h1);
    put(h0, h, mul(k.A0, shell_weight(h, rho58)));
  }
#pragma unroll 1
  for (int j = 0; j < axis; ++j) {
    if (!(mask >> (1 + j) & 1u)) continue;
    const ShellInfo& h = c.shell[1 + j];
    pre(h, h4);
    const Factor w = shell_weight(h, rho58);
    const int a = h.a, n = a * a;
    i64 sym = k.A0 + n * k.A1, anti = k.P0, x = k.Rx0, y = k.Ry0;
    if (S::ORDER >= 4) {
      sym += (n * n) * k.A2;
      anti += n * k.P1;
    }
    if (S::ORDER >= 3) {
      x += n * (k.Rx1 + k.Tx);
      y += n * (k.Ry1 + k.Ty);
    }
    x *= a;
    y *= a;
    anti *= n;
    put(h0, h, mul(sym + anti + x, w));
    put(h1, h, mul(sym - anti + y, w));
    put(h2, h, mul(sym + anti - x, w));
    put(h3, h, mul(sym - anti - y, w));
  }
#pragma unroll 1
  for (int j = 0; j < diag; ++j) {
    if (!(mask >> (1 + axis + j) & 1u)) continue;
    const ShellInfo& h = c.shell[1 + axis + j];
    pre(h, h4);
    const Factor w = shell_weight(h, rho58);
    const int a = h.a, a2 = a * a, n = 2 * a2;
    i64 sym = k.A0 + n * k.A1, cross = k.Q0, x = k.Rx0, y = k.Ry0;
    if (S::ORDER >= 4) {
      sym += (n * n) * k.A2 + (a2 * a2) * k.B;
      cross += n * k.Q1;
    }
    if (S::ORDER >= 3) {
      x += n * k.Rx1 + a2 * k.Tx;
      y += n * k.Ry1 + a2 * k.Ty;
    }
    cross *= a2;
    x *= a;
    y *= a;
    const i64 p = sym + cross, m = sym - cross, u = x + y, v = y - x;
    put(h0, h, mul(p + u, w));
    put(h1, h, mul(m + v, w));
    put(h2, h, mul(p - u, w));
    put(h3, h, mul(m - v, w));
  }
#pragma unroll 1
  for (int j = 0; j < octet; ++j) {
    if (!(mask >> (1 + axis + diag + j) & 1u)) continue;
    const ShellInfo& h = c.shell[1 + axis + diag + j];
    pre(h, h8);
    const Factor w = shell_weight(h, rho58);
    const int a = h.a, b = h.b, a2 = a * a, b2 = b * b, ab = a * b, n = a2 + b2, d = a2 - b2;
    const i64 sym = k.A0 + n * k.A1 + (n * n) * k.A2 + (ab * ab) * k.B;
    const i64 anti = d * (k.P0 + n * k.P1), q = ab * (k.Q0 + n * k.Q1), q2 = (ab * d) * k.Q2;
    const i64 ux = k.Rx0 + n * k.Rx1, uy = k.Ry0 + n * k.Ry1;
    {   // |e_x| = a, |e_y| = b: directions 0 and 3 and their opposites 4 and 7
      const i64 x = a * (ux + a2 * k.Tx), y = b * (uy + b2 * k.Ty);
      const i64 p = sym + anti + q + q2, m = sym + anti - q - q2;
      put(h0, h, mul(p + x + y, w));
      put(h3, h, mul(m - x + y, w));
      put(h4, h, mul(p - x - y, w));
      put(h7, h, mul(m + x - y, w));
    }
    {   // |e_x| = b, |e_y| = a: 1, 2 and 5, 6
      const i64 x = b * (ux + b2 * k.Tx), y = a * (uy + a2 * k.Ty);
      const i64 p = sym - anti + q - q2, m = sym - anti - q + q2;
      put(h1, h, mul(p + x + y, w));
      put(h2, h, mul(m - x + y, w));
      put(h5, h, mul(p - x - y, w));
      put(h6, h, mul(m + x - y, w));
    }
  }
}

// Lattice velocity of direction `first + h` of a shell (for the few nodes that need it).
LBM_HD void velocity(const ShellInfo& s, int h, int& ex, int& ey) {
  const int a = s.a, b = s.b;
  if (a == 0) {
    ex = ey = 0;
  } else if (b == 0) {
    ex = h == 0 ? a : h == 2 ? -a : 0;
    ey = h == 1 ? a : h == 3 ? -a : 0;
  } else if (a == b) {
    ex = h == 0 || h == 3 ? a : -a;
    ey = h < 2 ? a : -a;
  } else {
    const int kx = h == 0 || h == 3 || h == 4 || h == 7 ? a : b;
    ex = h < 2 || h > 5 ? kx : -kx;
    ey = h < 4 ? a + b - kx : -(a + b - kx);
  }
}

// Moments of a node's populations: rho, sum f e_x, sum f e_y, sum f |e|^2 (times 2^-E), in
// units of 2^-58. Each shell is summed exactly (at most eight values below 2^59) and then
// rounded to the common unit, which the shells up to weight 2^-4 are multiples of near rest (a
// half rounds up: the fewer halves, the less bias).
struct Moments {
  i64 rho, jx, jy, e2;
};

// Reads a node's doubles at f[i * stride], leaves their integers there and sums them (the shells in
// `mask`); `low` as in load().
template <class S>
LBM_HD Moments gather(const Consts& c, double* f, int stride, int& low,
                      unsigned mask = kAllShells) {
  constexpr int axis = kind_count<S>(1), diag = kind_count<S>(2), octet = kind_count<S>(3);
  auto get = [&](const ShellInfo& s, int h) {
    double* at = f + (s.first + h) * stride;
    const i64 F = load(*at, s.fe, c.E, low);
    *at = double_of((u64)F);
    return F;
  };
  Moments m{0, 0, 0, 0};
  auto add = [&](const ShellInfo& s, int n, i64 sum, i64 x, i64 y) {
    const int sh = s.fe - 58;
    const i64 half = (1ll << sh) >> 1;
    sum = (sum + half) >> sh;
    m.rho += sum;
    m.jx += (x + half) >> sh;
    m.jy += (y + half) >> sh;
    m.e2 += n * sum;
  };
  if (mask & 1u) {
    const ShellInfo& s = c.shell[0];
    m.rho = get(s, 0) << (58 - s.fe);   // the rest weight is above 1/8: fe = 56 or 57
  }
#pragma unroll 1
  for (int j = 0; j < axis; ++j) {
    if (!(mask >> (1 + j) & 1u)) continue;
    const ShellInfo& s = c.shell[1 + j];
    const i64 p0 = get(s, 0), p1 = get(s, 1), p2 = get(s, 2), p3 = get(s, 3);
    add(s, s.a * s.a, p0 + p1 + p2 + p3, s.a * (p0 - p2), s.a * (p1 - p3));
  }
#pragma unroll 1
  for (int j = 0; j < diag; ++j) {
    if (!(mask >> (1 + axis + j) & 1u)) continue;
    const ShellInfo& s = c.shell[1 + axis + j];
    const i64 p0 = get(s, 0), p1 = get(s, 1), p2 = get(s, 2), p3 = get(s, 3);
    add(s, 2 * s.a * s.a, p0 + p1 + p2 + p3, s.a * (p0 - p1 - p2 + p3), s.a * (p0 + p1 - p2 - p3));
  }
#pragma unroll 1
  for (int j = 0; j < octet; ++j) {
    if (!(mask >> (1 + axis + diag + j) & 1u)) continue;
    const ShellInfo& s = c.shell[1 + axis + diag + j];
    const i64 p0 = get(s, 0), p1 = get(s, 1), p2 = get(s, 2), p3 = get(s, 3);
    const i64 p4 = get(s, 4), p5 = get(s, 5), p6 = get(s, 6), p7 = get(s, 7);
    const i64 d0 = p0 - p4, d1 = p1 - p5, d2 = p2 - p6, d3 = p3 - p7;
    add(s, s.a * s.a + s.b * s.b, ((p0 + p1) + (p2 + p3)) + ((p4 + p5) + (p6 + p7)),
        s.a * (d0 - d3) + s.b * (d1 - d2), s.b * (d0 + d3) + s.a * (d1 + d2));
  }
  return m;
}

// 1 / v for 1/2 < v < 2, both in units of 2^-60: from the single-precision reciprocal x of the
// leading bits, x (1 + e + e^2) with e = 1 - v x (the geometric series; e^3 < 2^-63 is left out).
LBM_HD i64 reciprocal(i64 v) {
  constexpr float kScale = 72057594037927936.0f;   // 2^56
#ifdef __CUDA_ARCH__
  const float f = __fdividef(kScale, (float)(int)(v >> 32));
#else
  const float f = kScale / (float)(int)(v >> 32);
#endif
  const Limbs x = split((i64)(int)f << 32);
  const i64 e = (1ll << 60) - prod(split(v), x);
  const Limbs es = split(e);
  return ((i64)x.h << 32) + prod(x, split(e + prod(es, es)));
}

// The shells of a stencil for given weights (w: one per direction); false if one lies outside the
// weights' range.
template <class S>
inline bool make_shells(const double* w, ShellInfo (&out)[8]) {
  int n = 0;
  for (int kind = 0; kind < 4; ++kind)
    for (int s = 0; s < S::NSHELL; ++s) {
      if (kind_of<S>(s) != kind) continue;
      int e;
      const double m = std::frexp(w[S::shell_first(s)], &e);   // w = m 2^e, m in [1/2, 1)
      if (!(m > 0.5) || e > 0 || e < -40) return false;
      out[n++] = ShellInfo{S::shell_first(s), S::shell_a(s), S::shell_b(s), 55 - e,
                           factor((i64)std::ldexp(m, 62))};
    }
  return true;
}

// 1/2 < rho 2^-E < 2, |(X, Y)|^2 <= 0.7, |T - 1| <= 1/4, for components and T - 1 known to be
// below 2
LBM_HD bool in_range(const State& u) {
  const i64 top = (i64)(0.7 * (double)(1ll << 60)), quarter = 1ll << 58;
  const Limbs X = split(u.X), Y = split(u.Y);
  return u.rho > (1ll << 57) && u.rho < (1ll << 59) && prod(X, X) + prod(Y, Y) <= top &&
         u.th <= quarter && u.th >= -quarter;
}

LBM_HD bool state(const Moments& m, const Consts& c, State& u) {
  // |sum f e| < rho and sum f |e|^2 < 4 rho hold well beyond the range and keep the quotients small
  if (m.rho <= (1ll << 57) || m.rho >= (1ll << 59) || m.jx >= m.rho || -m.jx >= m.rho ||
      m.jy >= m.rho || -m.jy >= m.rho || m.e2 >= 4 * m.rho)
    return false;
  const Limbs ri = split(prod(c.r2, split(reciprocal(m.rho << 2))));
  u.rho = m.rho;
  u.X = prod(split(m.jx << 2), ri);
  u.Y = prod(split(m.jy << 2), ri);
  // D rho T = r^2 sum f |e|^2 - rho u^2 with D = 2 and u = (X, Y) / r
  const Limbs X = split(u.X), Y = split(u.Y);
  const i64 u2 = prod(split(prod(X, X) + prod(Y, Y)), c.inv_r2);
  u.th = prod(split(m.e2 << 1), ri) - (u2 >> 1) - (1ll << 60);
  return in_range(u);
}

// The state of given density, r u and temperature; false out of the range.
LBM_HD bool state_of(double rho, double X, double Y, double T, const Consts& c, State& u) {
  const double p = rho * pow2(-c.E), th = T - 1.0;
  if (!(p < 2.0 && p > 0.5 && fabs(X) < 2.0 && fabs(Y) < 2.0 && fabs(th) < 2.0)) return false;
  u.rho = fixed60(p) >> 2;
  u.X = fixed60(X);
  u.Y = fixed60(Y);
  u.th = fixed60(th);
  return in_range(u);
}

}  // namespace fx
}  // namespace lbm
