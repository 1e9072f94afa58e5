// The FP64 collision of collide.cuh evaluated in 64-bit fixed point, on the integer and FP32 pipes.
//
// Why: GB300 issues two FP64 lanes per SM and clock, 1/64 of its integer and FP32 rate, so the
// about 400 FP64 instructions of a collision take 64 issue slots each and the FP64 pipe alone sets
// the time of an FP64 step (17 times its DRAM time).  In fixed point relative to the node's
// largest population the sums are exact, the products are four 32-bit multiplications,
// and only the quotient kappa takes (FP32) floating point, refined by integer remainders.
// Measured per step: 96 x 80 x 72 plume 0.511 -> 0.16 ms, 128^3 with tensor field and source 1.80 ->
// 0.59 ms, the first steps of a 128^3 plume 2.1 -> 0.72 ms.  What bounds it now is instruction issue
// (6800 per warp, 56 % of the slots) with 12 warps per SM, at 0.18 of the DRAM rate.  Steep tails are
// left to FP64 (collide64.cuh), where they make up most of a box at little gain: the 256^3 plume 8
// nodes wide takes 13.1 to 17.7 ms a step where FP64 arithmetic takes 17.8 to 20.1.
//
// Representation: population i is held as 4^n_i g_i, n_i its number of nonzero velocity components
// (all of them about 8/27 phi near equilibrium, W_i = 8/27 4^-n_i), in units U = 2^(etop - 57),
// etop the exponent of the largest.  So t = max 4^n_i |g_i| < 2^58 U, and with
// sum 4^-n_i = 27/8 every intermediate stays below 2^63:
//     S = sum |g_i| <= 3.4 t,  |m_a| <= 1.2 t,  |j_a| <= 2.5 t,  |(T - I) j| <= |j|,
//     8/9 |c.(a - j)| <= 14 t < 2^62.
// U is 1e-18 to 3e-18 of phi near equilibrium, a tenth of the FP64 rounding of the rest population,
// so the result (rounded to FP64 once, at the end) is closer to the exact collision than FP64
// arithmetic gives.  Populations below t/32 lose the bits under the unit; where that would tell in the
// others, in the fallback's alpha, they are read again (blend_given).
//
// With 3 W_i = (8/9) 4^-n_i, and m = sum c g = j + phi u,
//     4^n b_i  = 4^n (phi E_i + 3 W_i c.j) = 8/27 phi (1 - 1.5 u.u + 4.5 (c.u)^2) + c.(8/9 m),
//     dh_i = g_i - b_i,
//     4^n g*_i = 4^n g_i + c.(8/9 (a - j)) - (1 + kappa) 4^n dh_i,
// and the rest population takes what the rounding of the others leaves of phi, so that the
// collision conserves the node's mass.
//
// collide_fixed refuses a node that this cannot hold as well as FP64 does (non-finite or extreme
// values, phi small beside the largest 4^n_i g_i, a correction larger than the node): the caller then
// pulls it again and runs the FP64 collision.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#include "lattice.cuh"

#ifdef __CUDACC__
#define ELBM_HD __host__ __device__ __forceinline__
#define ELBM_COLD __host__ __device__ __noinline__
#else
#define ELBM_HD inline
#define ELBM_COLD inline
#endif

namespace elbm {

// A number |c| < 1/2 as h 2^-32 + l 2^-64 with signed 32-bit h and l; as well the digits of an
// integer h 2^32 + l.
struct Q64 {
  int32_t h, l;
};
ELBM_HD Q64 digits(int64_t x) { return Q64{(int32_t)((x + 0x80000000ll) >> 32), (int32_t)x}; }

// x c rounded to the nearest unit: four multiplications and two additions on 32-bit digits.
ELBM_HD int64_t mulq(Q64 x, Q64 c) {
  const int64_t w = (int64_t)x.l * c.h + ((int64_t)x.h * c.l + 0x80000000ll);
  return (int64_t)x.h * c.h + (int32_t)(w >> 32);
}
ELBM_HD int64_t mulq(int64_t x, Q64 c) { return mulq(digits(x), c); }

// Per-launch constants (host): the equilibrium polynomial times the rest weight 8/27, and the
// stabilizer's tables.
struct FixConsts {
  Q64 base;        // 8/27 (1 - 1.5 u.u)
  Q64 quad[6];     // 8/27 4.5 (ux ux, 2 ux uy, 2 ux uz, uy uy, 2 uy uz, uz uz)
  Q64 u[3];
  Q64 TmI[6];      // (T - I) / 4 of the uniform T = 2I - S
  Q64 K3[Q], L[Q], M[Q];   // 4^-n K3 / 8, 4^-n L, 16^-n M / 16
  uint32_t exponent[Q];    // (5 - 2 n) << 20 (from_fixed)
  double E[Q];
  double theta2;
  bool ok;                 // the tables fit, and the positivity threshold is 0
};

inline Q64 q64_host(long double v) {
  return digits((int64_t)(v * 18446744073709551616.0L + (v >= 0 ? 0.5L : -0.5L)));
}

// From the FP64 tables of PopConsts<double>.
template <typename Consts>
inline FixConsts fix_consts(const Consts& k) {
  FixConsts f;
  const long double u[3] = {k.ux, k.uy, k.uz}, w0 = 8.0L / 27.0L;
  f.base = q64_host(w0 * (1.0L - 1.5L * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])));
  const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
  f.ok = k.eps == 0;
  for (int a = 0; a < 3; ++a) f.ok = f.ok && std::fabs((double)u[a]) < 0.4;
  if (!f.ok) return f;
  for (int q = 0; q < 6; ++q) f.quad[q] = q64_host(w0 * 4.5L * (ia[q] == ib[q] ? 1.0L : 2.0L) * u[ia[q]] * u[ib[q]]);
  for (int a = 0; a < 3; ++a) f.u[a] = q64_host(u[a]);
  const long double T[6] = {k.T.xx - 1.0L, k.T.xy, k.T.xz, k.T.yy - 1.0L, k.T.yz, k.T.zz - 1.0L};
  for (int q = 0; q < 6; ++q) f.ok = f.ok && std::fabs((double)T[q]) < 1.5;   // not so where T is not finite
  if (!f.ok) return f;
  for (int q = 0; q < 6; ++q) f.TmI[q] = q64_host(0.25L * T[q]);
  for (int i = 0; i < Q; ++i) {
    const long double s = 1.0L / (1 << (2 * nnz_of(i)));   // of 4^n dh_i
    f.ok = f.ok && std::fabs(k.K3[i]) < 3.9 && std::fabs(k.L[i]) < 0.4 && s * s * k.M[i] < 7.9L;
    if (!f.ok) return f;
    f.K3[i] = q64_host(0.125L * s * k.K3[i]);
    f.L[i] = q64_host(s * k.L[i]);
    f.M[i] = q64_host(0.0625L * s * s * k.M[i]);
    f.exponent[i] = (uint32_t)(5 - 2 * nnz_of(i)) << 20;
    f.E[i] = k.E[i];
  }
  f.theta2 = k.theta2;
  return f;
}

ELBM_HD uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return b;
#endif
}
ELBM_HD double value_of(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
ELBM_HD int clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}
ELBM_HD int clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return __builtin_clz(v);
#endif
}
ELBM_HD float pow2f(int n) {   // -126 <= n <= 127
  const uint32_t b = (uint32_t)(n + 127) << 23;
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float v;
  memcpy(&v, &b, 4);
  return v;
#endif
}
ELBM_HD float quotient(float a, float b) {   // to a few units in the last place
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return a / b;
#endif
}

// 4^n |v| in units 2^(etop - 57), for 4^n |v| < 2^(etop + 1) (etop: biased exponent); values below
// t/32 lose the bits under the unit.
ELBM_HD int64_t to_fixed(uint64_t b, int n, int etop) {
  const int e = ((int)(b >> 52) & 0x7ff) + 2 * n;
  const int d = etop - e < 63 ? etop - e : 63;       // zero and subnormals shift out
  return (int64_t)((((b & 0xfffffffffffffull) | 0x10000000000000ull) << 5) >> d);
}

// v/4 in units 2^-64, for |v| < 2.
ELBM_HD int64_t to_quarter(double v) {
  const uint64_t b = bits_of(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const int d = 1023 - e < 63 ? 1023 - e : 63;
  const int64_t x = (int64_t)((((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) >> d);
  return (int64_t)b < 0 ? -x : x;
}

// 4^-n m units of 2^(etop - 57) as FP64, rounded to nearest even, with the sign bit `neg` (bit 31).
// e: (etop - 2 n - 57 + 62) << 20.
ELBM_HD double from_fixed(uint64_t m, uint32_t neg, uint32_t e) {
  const int z = clz64(m | 1);                         // >= 1
  const uint64_t t = m << (z - 1);                    // leading bit at 62
  const uint64_t q = (t + 0x1ff + ((t >> 10) & 1)) >> 10;
  // q holds the leading bit at 52 (or 53 after a carry), which adds 1 to the exponent field
  uint32_t hi = (uint32_t)(q >> 32) + e - ((uint32_t)z << 20);
  hi = m == 0 ? 0u : hi | neg;
  return value_of((uint64_t)hi << 32 | (uint32_t)q);
}

// den 2^(68 - 2 sh) > theta^2 phi^2, in FP32 unless the two are within its rounding.
ELBM_HD bool above_guard(int64_t den, int64_t phi, int sh, double theta2) {
  const float f = (float)phi, a = (float)den, b = (float)theta2 * f * (f * pow2f(2 * sh - 68));
  if (fabsf(a - b) > 1e-5f * b) return a > b;
  const double p = (double)phi * (double)(1ull << sh);
  return (double)den * 0x1p68 > theta2 * (p * p);
}

// The 13 velocities whose first nonzero component is positive are those of i = 14 .. 26; their
// c.v, v an integer vector.
ELBM_HD void dots13(int64_t x, int64_t y, int64_t z, int64_t (&d)[13]) {
  const int64_t p = y + z, q = y - z;
  d[0] = z;
  d[1] = q;
  d[2] = y;
  d[3] = p;
  d[4] = x - p;
  d[5] = x - y;
  d[6] = x - q;
  d[7] = x - z;
  d[8] = x;
  d[9] = x + z;
  d[10] = x + q;
  d[11] = x + y;
  d[12] = x + p;
}

// phi times the even part of the equilibrium polynomial (and the rest weight) for those 13.
ELBM_HD void evens13(int64_t A, const int64_t (&B)[6], int64_t (&e)[13]) {
  const int64_t ax = A + B[0], ay = A + B[3], az = A + B[5];
  const int64_t yz = ay + B[5], xy = ax + B[3], xz = ax + B[5], xyz = xy + B[5];
  const int64_t p = B[1] + B[2], q = B[1] - B[2];
  const int64_t s = xyz + B[4], t = xyz - B[4];
  e[0] = az;
  e[1] = yz - B[4];
  e[2] = ay;
  e[3] = yz + B[4];
  e[4] = s - p;       // (1, -1, -1): -Bxy - Bxz + Byz
  e[5] = xy - B[1];
  e[6] = t - q;       // (1, -1, 1): -Bxy + Bxz - Byz
  e[7] = xz - B[2];
  e[8] = ax;
  e[9] = xz + B[2];
  e[10] = t + q;      // (1, 1, -1): Bxy - Bxz - Byz
  e[11] = xy + B[1];
  e[12] = s + p;
}

// s0 + s1/4 + s2/16 + s3/64, to the nearest.
ELBM_HD int64_t weigh(int64_t s0, int64_t s1, int64_t s2, int64_t s3) {
  return s0 + ((s1 + ((s2 + ((s3 + 2) >> 2) + 2) >> 2) + 2) >> 2);
}

// sum g_i from the 4^n g_i.
ELBM_HD int64_t mass_of(const int64_t (&G)[Q]) {
  int64_t c[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < Q; ++i) c[nnz_of(i)] += G[i];
  return weigh(c[0], c[1], c[2], c[3]);
}

// num / (2 den) in units of 2^-64 (scale 2^63 = 1/2), den > 0: three quotients of about 22 bits each with
// exact remainders in between; false where it is 1/4 or more.
ELBM_HD bool half_quotient(int64_t num, int64_t den, float limit, int64_t& out) {
  const float rd = quotient(1.0f, (float)den);
  const Q64 d = digits(den);
  int64_t rem = num, c = 0;
#pragma unroll
  for (int it = 0; it < 3; ++it) {
    const float q = (float)rem * rd * 0x1p63f;
    if (!(q < limit && q > -limit)) return false;
    const int64_t step = (int64_t)llrintf(q);
    c += step;
    rem -= 2 * mulq(d, digits(step));
  }
  out = c;
  return true;
}

// Where a node's integers are kept: G_i = 4^n g_i, X_i = first 4^n dh_i, then the result, and one
// number per pair of opposite velocities; in local arrays, or (fast) in shared memory, thread t's
// at p[i stride].
constexpr int KEPT = 2 * Q + 13;
struct InLocal {
  int64_t v[KEPT];
  ELBM_HD int64_t& g(int i) { return v[i]; }
  ELBM_HD int64_t& x(int i) { return v[Q + i]; }
  ELBM_HD int64_t& pair(int i) { return v[2 * Q + i]; }
};
template <int STRIDE>
struct InShared {
  int64_t* p;
  ELBM_HD int64_t& g(int i) { return p[i * STRIDE]; }
  ELBM_HD int64_t& x(int i) { return p[(Q + i) * STRIDE]; }
  ELBM_HD int64_t& pair(int i) { return p[(2 * Q + i) * STRIDE]; }
};

// What collide_fixed did with a node: left it to FP64, collided it, or came to a fallback whose alpha
// takes more bits than it kept (blend_given ends such a node).
enum class Fixed { REFUSED, DONE, SMALL_ALPHA };

// keep.x(i) from keep.g(i) towards keep.x(i) by alpha = 2^-63 half (far), or from keep.x(i) towards
// keep.g(i) by 1 - alpha = 2^-63 half.
template <typename Keep>
ELBM_HD void blend(Keep& keep, int64_t half, bool far) {
  const Q64 aq = digits(half > 0 ? half : 0);
#pragma unroll 1
  for (int i = 0; i < Q; ++i) {
    const int64_t gi = keep.g(i), x = keep.x(i), m = mulq(2 * (gi - x), aq), b = far ? gi - m : x + m;
    // the deciding population becomes 0, not a unit below: whole units of opposite sign meet and
    // cancel where a plume's surroundings are empty, and 1/phi then overflows
    keep.x(i) = gi >= 0 && b < 0 ? 0 : b;
  }
}

// The results keep.x to out(i, value).
template <typename Keep, typename Out>
ELBM_HD void put(Keep& keep, int etop, const FixConsts& k, Out& out) {
#pragma unroll 3
  for (int i = 0; i < Q; ++i) {
    const int64_t x = keep.x(i);
    out(i, from_fixed((uint64_t)(x < 0 ? -x : x), (uint32_t)(x >> 32) & 0x80000000u, k.exponent[i] + ((uint32_t)etop << 20)));
  }
}

// The fallback of a node whose deciding d is less than 1/16 of the largest: a unit of its g moves the
// other populations by more than 16 units, where FP64 arithmetic knows a g that is small beside the
// others to its last bit.  So alpha is formed in FP64 from given(i), population i as collide_fixed got
// it, with its source.  Out of line and ended here: with its loop in collide_fixed the step of the
// driven 128^3 box, which never comes here, took 12.5 instead of 7.7 ms (12 steps and read-outs).
template <typename Keep, typename Out, typename Given>
ELBM_COLD void blend_given(Keep& keep, int etop, const FixConsts& k, Out out, Given given) {
  // Only populations whose kept digits leave it open decide; the others need not be fetched again.
  float most = 1.0f;
#pragma unroll 1
  for (int i = 0; i < Q; ++i) {
    const int64_t gi = keep.g(i), x = keep.x(i);
    if (x < 0 && gi > x) most = fminf(most, quotient((float)(gi > 0 ? gi : 0) + 2.0f, (float)(gi - x)));
  }
  most *= 1.001f;
  const double unit = value_of((uint64_t)(2103 - etop) << 52);
  double num = 1.0, den = 1.0;                        // alpha
#pragma unroll 1
  for (int i = 0; i < Q; ++i) {
    const int64_t gi = keep.g(i), x = keep.x(i);
    if (x < 0 && gi > x && (float)gi - 2.0f <= most * ((float)(gi - x) + 2.0f)) {
      const double g = given(i), n = g > 0.0 ? g * (double)(1 << (2 * nnz_of(i))) * unit : 0.0, d = n - (double)x;
      if (n * den < num * d) {
        num = n;
        den = d;
      }
    }
  }
  const bool far = num < 0.5 * den;
  blend(keep, (int64_t)((far ? num : den - num) / den * 0x1p63), far);
  put(keep, etop, k, out);
}

// One node.  v: the 27 pre-collision populations.  Tn: the node's T, or null for the uniform one.
// src: source term r, g_i + r E_i is collided (0: none).  keep: storage for the node's integers.
// out(i, value): receives the post-collision populations (only of a node that is DONE).
// took: the positivity fallback (threshold 0) was taken.  etop: what blend_given needs besides keep.
// vote(refuse): whether the node is refused, where it would be by itself or not.
//
// The loops with products and conversions are not unrolled: unrolled, the collision is about 90 KB
// of instructions that every warp runs through once, and fetching them, not executing them, sets
// the pace (ncu: 2.6 to 4.6 warps per issue stalled for want of instructions).
template <int VEL, typename Keep, typename Out, typename Vote>
ELBM_HD Fixed collide_fixed(const double (&v)[Q], const double* Tn, double src, bool has_src, bool fallback,
                            const FixConsts& k, Keep& keep, bool& took, int& etop, Out out, Vote vote) {
  took = false;
  uint32_t top = 0, sign = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const uint32_t h = (uint32_t)(bits_of(v[i]) >> 32);
    const uint32_t a = (h & 0x7fffffffu) + ((uint32_t)nnz_of(i) << 21);
    top = a > top ? a : top;
    sign |= h;
  }
  if (has_src) {
    const uint32_t h = (uint32_t)(bits_of(src) >> 32), a = h & 0x7fffffffu;
    top = a > top ? a : top;
    sign |= h;
  }
  etop = (int)(top >> 20);
  bool refuse = etop < 150 || etop > 1900;           // also inf and NaN
  const Q64 c49{1908874354, -954437177};             // 4/9
  int64_t phi, mx, my, mz;
  {
    int64_t G[Q], d[13];
#pragma unroll
    for (int i = 0; i < Q; ++i) G[i] = to_fixed(bits_of(v[i]), nnz_of(i), etop);
    if ((int32_t)sign < 0) {
#pragma unroll
      for (int i = 0; i < Q; ++i) G[i] = (int64_t)bits_of(v[i]) < 0 ? -G[i] : G[i];
    }
    if (has_src) {
      // r E_i = r W_i (1 - 1.5 u.u + 4.5 (c.u)^2 + 3 c.u)
      const int64_t rm = to_fixed(bits_of(src), 0, etop), r = (int64_t)bits_of(src) < 0 ? -rm : rm;
      const int64_t A = mulq(r, k.base);
      if (VEL == 0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) G[i] += A;
      } else {
        const int64_t r89 = mulq(2 * r, c49);
        int64_t B[6], e[13];
#pragma unroll
        for (int q = 0; q < 6; ++q) B[q] = mulq(r, k.quad[q]);
        evens13(A, B, e);
        dots13(mulq(r89, k.u[0]), mulq(r89, k.u[1]), mulq(r89, k.u[2]), d);
        G[13] += A;
#pragma unroll
        for (int i = 14; i < Q; ++i) {
          G[i] += e[i - 14] + d[i - 14];
          G[26 - i] += e[i - 14] - d[i - 14];
        }
      }
    }
    // moments, by classes of 1, 2 and 3 nonzero components (d: the odd part of each pair)
#pragma unroll
    for (int i = 14; i < Q; ++i) d[i - 14] = G[i] - G[26 - i];
    phi = mass_of(G);
    mx = weigh(0, d[8], (d[5] + d[11]) + (d[7] + d[9]), (d[4] + d[6]) + (d[10] + d[12]));
    my = weigh(0, d[2], (d[1] + d[3]) + (d[11] - d[5]), (d[10] - d[4]) + (d[12] - d[6]));
    mz = weigh(0, d[0], (d[3] - d[1]) + (d[9] - d[7]), (d[6] - d[4]) + (d[12] - d[10]));
    // phi below t/8 to t/4: the units would be coarse beside it
    refuse |= phi < (1ll << 55);
    if (VEL != 0 && (int32_t)sign < 0) {
      int64_t c[4] = {0, 0, 0, 0};
#pragma unroll
      for (int i = 0; i < Q; ++i) c[nnz_of(i)] -= G[i] < 0 ? G[i] : 0;
      refuse |= phi < (weigh(c[0], c[1], c[2], c[3]) >> 3);
    }
    // nearly all refusals are known here, at a tenth of the collision's instructions
    if (vote(refuse)) return Fixed::REFUSED;
    if (VEL != 0 || fallback) {
#pragma unroll
      for (int i = 0; i < Q; ++i) keep.g(i) = G[i];
    }
    if (VEL != 0) {
      // X: 4^n dh
      const Q64 f = digits(phi);
      int64_t B[6], e[13];
#pragma unroll
      for (int q = 0; q < 6; ++q) B[q] = mulq(f, k.quad[q]);
      const int64_t A = mulq(f, k.base);
      evens13(A, B, e);
      dots13(mulq(2 * mx, c49), mulq(2 * my, c49), mulq(2 * mz, c49), d);
      keep.x(13) = G[13] - A;
#pragma unroll
      for (int i = 14; i < Q; ++i) {
        keep.x(i) = G[i] - (e[i - 14] + d[i - 14]);
        keep.x(26 - i) = G[26 - i] - (e[i - 14] - d[i - 14]);
      }
    }
  }
  int64_t jx = mx, jy = my, jz = mz;
  if (VEL != 0) {
    const Q64 f = digits(phi);
    jx -= mulq(f, k.u[0]);
    jy -= mulq(f, k.u[1]);
    jz -= mulq(f, k.u[2]);
  }
  // a = (T - I) j
  int64_t ax, ay, az;
  {
    if (Tn != nullptr) {
      // T = 2I - S < 2, but rounds to 2 and a little above for D of 5e14 and more
      uint32_t any = 0;
#pragma unroll
      for (int q = 0; q < 6; ++q) any |= (uint32_t)(bits_of(Tn[q]) >> 32);
      if ((any & 0x40000000u) != 0) return Fixed::REFUSED;   // the exponent of some |T| >= 2, or NaN
    }
    Q64 T[6];
#pragma unroll
    for (int q = 0; q < 6; ++q)
      T[q] = Tn == nullptr ? k.TmI[q] : digits(to_quarter(Tn[q]) - (q == 0 || q == 3 || q == 5 ? 1ll << 62 : 0));
    const Q64 x = digits(4 * jx), y = digits(4 * jy), z = digits(4 * jz);
    ax = mulq(x, T[0]) + mulq(y, T[1]) + mulq(z, T[2]);
    ay = mulq(x, T[1]) + mulq(y, T[3]) + mulq(z, T[4]);
    az = mulq(x, T[2]) + mulq(y, T[4]) + mulq(z, T[5]);
  }
  int64_t any = 0, d[13];
  if (VEL == 0) {
    const int64_t A = mulq(phi, k.base);
    dots13(mulq(2 * ax, c49), mulq(2 * ay, c49), mulq(2 * az, c49), d);
    // the odd parts cancel in the sums over the classes of 6, 12 and 8 populations
    int64_t rest = phi - weigh(0, 6 * A, 12 * A, 8 * A);
    any = rest;
    keep.x(13) = rest;
#pragma unroll
    for (int i = 14; i < Q; ++i) {
      const int64_t p = A + d[i - 14], m = A - d[i - 14];
      keep.x(i) = p;
      keep.x(26 - i) = m;
      any |= p | m;
    }
  } else {
    // |4^n dh| < 2^62 after a shift up by sh, 2 <= sh <= 30
    uint32_t mag = 0;
#pragma unroll 3
    for (int i = 0; i < Q; ++i) {
      const int64_t x = keep.x(i);
      mag |= (uint32_t)((int32_t)(x >> 32) ^ (int32_t)(x >> 63));
    }
    if (mag >= 1u << 28) return Fixed::REFUSED;
    const int sh = mag == 0 ? 30 : clz32(mag) - 2;
    // kappa 2^-sh = num / (2 den), num = sum dh (K3 c.a + L phi) / 8, den = sum dh^2 M / 16
    int64_t Vx = 0, Vy = 0, Vz = 0, w, den;
    {
      const Q64 x = digits((int64_t)((uint64_t)keep.x(13) << sh));
      w = mulq(x, k.L[13]);
      den = mulq(mulq(x, x), k.M[13]);
    }
#pragma unroll 1
    for (int i = 14; i < Q; ++i) {
      const Q64 p = digits((int64_t)((uint64_t)keep.x(i) << sh));
      const Q64 m = digits((int64_t)((uint64_t)keep.x(26 - i) << sh));
      keep.pair(i - 14) = mulq(p, k.K3[i]) - mulq(m, k.K3[26 - i]);
      w += mulq(p, k.L[i]) + mulq(m, k.L[26 - i]);
      den += mulq(mulq(p, p), k.M[i]) + mulq(mulq(m, m), k.M[26 - i]);
    }
#pragma unroll
    for (int i = 14; i < Q; ++i) {
      const int64_t y = keep.pair(i - 14);
      Vx += cx_of(i) > 0 ? y : 0;
      Vy += cy_of(i) == 0 ? 0 : (cy_of(i) > 0 ? y : -y);
      Vz += cz_of(i) == 0 ? 0 : (cz_of(i) > 0 ? y : -y);
    }
    // (1 + kappa) 2^-sh in units of 2^-64; the 1 exactly
    int64_t c = 1ll << (64 - sh);
    if (above_guard(den, phi, sh, k.theta2)) {
      // a and w shifted up, so that the products keep their bits
      const uint64_t am = (uint64_t)(ax ^ (ax >> 63)) | (uint64_t)(ay ^ (ay >> 63)) | (uint64_t)(az ^ (az >> 63)) |
                          (uint64_t)(w ^ (w >> 63));
      const int sa = am >> 57 != 0 ? 0 : (clz64(am) - 6 < 24 ? clz64(am) - 6 : 24);
      const int64_t num = mulq((int64_t)((uint64_t)ax << sa), digits(Vx)) + mulq((int64_t)((uint64_t)ay << sa), digits(Vy)) +
                          mulq((int64_t)((uint64_t)az << sa), digits(Vz)) +
                          mulq((int64_t)((uint64_t)w << sa), digits(phi >> 3));
      int64_t kap;                                     // kappa 2^(sa - sh)
      if (!half_quotient(num, den, 0x1.fffep61f, kap)) return Fixed::REFUSED;   // c below 2^63 - 2^43, sh >= 2
      c += sa == 0 ? kap : (kap + (1ll << (sa - 1))) >> sa;
    }
    const Q64 cq = digits(c);
    dots13(mulq(2 * (ax - jx), c49), mulq(2 * (ay - jy), c49), mulq(2 * (az - jz), c49), d);
#pragma unroll
    for (int i = 0; i < 13; ++i) keep.pair(i) = d[i];
#pragma unroll 1
    for (int i = 14; i < Q; ++i) {
      const int64_t D = keep.pair(i - 14);
      const int64_t p = keep.g(i) + D - mulq((int64_t)((uint64_t)keep.x(i) << sh), cq);
      const int64_t m = keep.g(26 - i) - D - mulq((int64_t)((uint64_t)keep.x(26 - i) << sh), cq);
      keep.x(i) = p;
      keep.x(26 - i) = m;
      keep.pair(i - 14) = p + m;
      any |= p | m;
    }
    int64_t c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
    for (int i = 14; i < Q; ++i) {
      const int64_t t = keep.pair(i - 14);
      c1 += nnz_of(i) == 1 ? t : 0;
      c2 += nnz_of(i) == 2 ? t : 0;
      c3 += nnz_of(i) == 3 ? t : 0;
    }
    const int64_t rest = phi - weigh(0, c1, c2, c3);
    any |= rest;
    keep.x(13) = rest;
  }
  if (fallback && any < 0) {
    took = true;
    // alpha = min g_i / (g_i - g*_i) over g*_i < 0 < g_i - g*_i, capped to [0, 1].  The smallest
    // ratio is found in FP32 (15 bits and more of the leading words); where another one is as
    // close as that, by exact products.
    float best = 2.0f, second = 2.0f;
    int64_t nb = 1, db = 1;
    uint32_t mag = 0;
#pragma unroll 1
    for (int i = 0; i < Q; ++i) {
      const int64_t gi = keep.g(i), x = keep.x(i), dd = gi - x;
      const uint32_t size = (uint32_t)((int32_t)(dd >> 32) ^ (int32_t)(dd >> 63));
      mag = size > mag ? size : mag;
      if (x < 0 && dd > 0) {
        const int64_t n = gi > 0 ? gi : 0;
        const float q = quotient((float)(int32_t)(n >> 32), (float)(int32_t)(dd >> 32) + 1.0f);
        second = fminf(second, fmaxf(q, best));
        if (q < best) {
          best = q;
          nb = n;
          db = dd;
        }
      }
    }
    if (mag >= (1u << 30) - 1) return Fixed::REFUSED;   // 2 d and its digits stay below 2^63
    if (second <= best * 1.0002f || nb < (1ll << 46)) {
#pragma unroll 1
      for (int i = 0; i < Q; ++i) {
        const int64_t gi = keep.g(i), x = keep.x(i), dd = gi - x;
        if (x < 0 && dd > 0) {
          const int64_t n = gi > 0 ? gi : 0;
          if ((unsigned __int128)(uint64_t)n * (uint64_t)db < (unsigned __int128)(uint64_t)nb * (uint64_t)dd) {
            nb = n;
            db = dd;
          }
        }
      }
    }
    if ((uint32_t)(db >> 28) < mag) return Fixed::SMALL_ALPHA;
    // The blend starts at the nearer end, by the smaller one of alpha and 1 - alpha = -g*/d: half of
    // that is at most 1/4, where alpha / 2 with alpha near 1 would reach the 2^63 that no int64_t holds.
    const bool far = nb < db - nb;                    // alpha < 1/2: from g
    int64_t half = 0;
    if (!half_quotient(far ? nb : db - nb, db, 0x1.1p62f, half)) return Fixed::REFUSED;
    blend(keep, half, far);
  }
  put(keep, etop, k, out);
  return Fixed::DONE;
}

// The whole collision where v still holds the populations as given; false for a node left to FP64.
template <int VEL, typename Keep, typename Out>
ELBM_HD bool collide_fixed(const double (&v)[Q], const double* Tn, double src, bool has_src, bool fallback,
                           const FixConsts& k, Keep& keep, bool& took, Out out) {
  int etop;
  const Fixed f = collide_fixed<VEL>(v, Tn, src, has_src, fallback, k, keep, took, etop, out,
                                     [](bool refuse) { return refuse; });
  if (f == Fixed::SMALL_ALPHA)
    blend_given(keep, etop, k, out, [&](int i) { return v[i] + (has_src ? src * k.E[i] : 0.0); });
  return f != Fixed::REFUSED;
}

}  // namespace elbm
