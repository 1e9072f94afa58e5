// Mass and entropy sums of the conservation diagnostics without FP64 arithmetic per population:
// sum v and sum v ln(v/W) (Eq. method-entropy) of the populations of a node (or a few nodes) in
// 64-bit fixed point relative to the largest of them, one FP64 addition per node.
//
// Why: GB300 issues two FP64 lanes per SM and clock, so the FP64 quotient and logarithm per
// population (about 25 FP64 instructions, 64 issue cycles each) set the time of a reduction, not
// DRAM.  The integer and FP32 pipes run at 64 times that rate; about 60 of their instructions
// replace those 25.
//
// A node's values are v = 2^e m, 1 <= m < 2, the largest of them has exponent etop, d = etop - e.
// In D dimensions with n nonzero velocity components -ln W = c0 + (2 n + 2) ln 2 with
// c0 = D ln 3 - (D + 2) ln 2, so that
//     ln(v/W) = (etop + 2) ln 2  +  (2 n - d) ln 2  +  (c0 + ln m),
// where the first term is the same for the whole node and the second and third are zero for the
// equilibrium of phi = 1 and velocity 0.  sum v, sum v (2 n - d) and sum v (c0 + ln m) are integer
// sums; their three products with constants are the node's only FP64 arithmetic.
//
// ln m: with c an integer near 4096/m, r = m c / 4096 - 1 is exact in integers (|r| < 2^-11), and
//     ln m = -ln(c/4096) + ln(1 + r),   ln(1 + r) = r - r^2/2 + r^3/3 - r^4/4 + r^5/5,
// with -ln(c/4096) from a table and r^3/3 - ... (below 2^-37) in FP32.  It is kept in units of
// 2^-62 with an error below 2^-59; the rounding of v/W alone costs an FP64 log(v/W) 2^-53.
#pragma once
#include <cstdint>
#include <type_traits>

namespace elbm {

constexpr double LN2 = 0.69314718055994530942, LN2_LOW = 2.3190468138462996e-17;   // their sum is ln 2
constexpr int LN_ENTRIES = 2049;   // c = 2048 .. 4096
// ln 2 and ln 3 in units of 2^-62
constexpr long long LN2_Q62 = 3196577161300663915ll, LN3_Q62 = 5066454931323234910ll;

// -ln(c/4096) * 2^62 for c = 2048 + k: sums of ln((j + 1)/j) = 2 artanh(1/(2j + 1)), by their
// series in units of 2^-100.
struct LnTable {
  long long v[LN_ENTRIES];
  constexpr LnTable() : v() {
    unsigned __int128 s = 0;
    v[LN_ENTRIES - 1] = 0;
    for (int c = 4095; c >= 2048; --c) {
      const unsigned __int128 n = 2 * (unsigned)c + 1;
      unsigned __int128 x = ((unsigned __int128)1 << 101) / n;
      for (int k = 1; k <= 9; k += 2) {
        s += x / k;
        x /= n * n;
      }
      v[c - 2048] = (long long)((s + ((unsigned __int128)1 << 37)) >> 38);
    }
  }
};

#ifdef __CUDACC__

static __device__ const LnTable g_ln_table = LnTable();

// The block's copy of the table with c0 added, for D dimensions (the caller synchronises
// afterwards).  c0 fits: c0 - ln(c/4096) lies in [-0.6, 0.6].
template <int D>
__device__ __forceinline__ void load_ln_table(long long (&t)[LN_ENTRIES]) {
  const unsigned long long c0 = (unsigned long long)D * LN3_Q62 - (unsigned long long)(D + 2) * LN2_Q62;
  for (int k = threadIdx.x + threadIdx.y * blockDim.x; k < LN_ENTRIES; k += blockDim.x * blockDim.y)
    t[k] = (long long)((unsigned long long)g_ln_table.v[k] + c0);
}

// r^3/3 - r^4/4 + r^5/5 in units of 2^-62, from rf = 4096 r.
__device__ __forceinline__ int ln1p_tail(float rf) {
  const float p = fmaf(rf, fmaf(rf, 0.8f, -4096.0f), 22369621.3f);
  return __float2int_rn(rf * rf * rf * p);
}

// c near 4096/m and, in cf, the same as a float (1 <= m < 2).
__device__ __forceinline__ unsigned ln_bin(float m, float& cf) {
  const float magic = 12582912.0f;   // 1.5 * 2^23: rounds to an integer in the low mantissa bits
  const float f = fmaf(__fdividef(1.0f, m), 4096.0f, magic);
  cf = f - magic;
  return __float_as_uint(f) & 0x1fffu;
}

// v (c0 + ln m) in units of 2^(e - 60), for v = 2^e m with mantissa man (m 2^23 or m 2^52).
__device__ __forceinline__ long long v_ln_m(uint32_t man, const long long (&t)[LN_ENTRIES]) {
  const float m = __uint_as_float(man + (126u << 23));   // man holds bit 23, which adds 1 to the exponent
  float cf;
  const unsigned c = ln_bin(m, cf);
  const int r = (int)(man * c);                          // r 2^35 (the 2^35 of m c drops out modulo 2^32)
  const float rf = fmaf(m, cf, -4096.0f);                // exact
  const long long s = (long long)r * r;                  // r^2 2^70
  const long long f = t[c - 2048] + ((long long)r << 27) - (s >> 9) + ln1p_tail(rf);
  const uint32_t h = man << 7;
  return (long long)(int)h * (int)(f >> 32) + __umulhi(h, (uint32_t)f);
}
__device__ __forceinline__ long long v_ln_m(uint64_t man, const long long (&t)[LN_ENTRIES]) {
  const float m = __uint_as_float(((uint32_t)(man >> 29) & 0x7fffffu) | 0x3f800000u);
  float cf;
  const unsigned c = ln_bin(m, cf);
  const long long r = (long long)(man * c);              // r 2^64
  const float rf = (float)(int)(r >> 30) * 0x1p-22f;
  const long long s = __mul64hi(r << 9, r << 9);         // r^2 2^82
  const long long f = t[c - 2048] + ((r + 2) >> 2) - (s >> 21) + ln1p_tail(rf);
  return __mul64hi((long long)(man << 10), f);
}

// The fields of a finite value: man (0 where the value is 0; FP32 subnormals count as 0, as in
// the kernels' arithmetic), e, and the sign.
__device__ __forceinline__ void split_value(float v, uint32_t& man, int& e, bool& neg) {
  const uint32_t b = __float_as_uint(v);
  const uint32_t x = (b >> 23) & 0xffu;
  man = x == 0u ? 0u : ((b & 0x7fffffu) | 0x800000u);
  e = (int)x - 127;
  neg = (b >> 31) != 0u;
}
__device__ __forceinline__ void split_value(double v, uint64_t& man, int& e, bool& neg) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int x = (int)(b >> 52) & 0x7ff;
  man = b & 0xfffffffffffffull;
  e = x - 1023;
  if (x != 0) {
    man |= 1ull << 52;
  } else if (man != 0) {               // subnormal: normalise
    const int sh = __clzll((long long)man) - 11;
    man <<= sh;
    e = -1022 - sh;
  }
  neg = (long long)b < 0;
}

// a 2^n
__device__ __forceinline__ double scaled(double a, int n) {
  return n < -1022 ? scalbn(a, n) : a * __hiloint2double((n + 1023) << 20, 0);
}

template <typename V>
__device__ __forceinline__ bool value_finite(V v) {
  return fabs(v) <= (sizeof(V) == 4 ? V(3.402823466e38f) : V(1.7976931348623157e308));
}

// entropy of a node from its integer sums: plus = sum v (units 2^(u - 3)), steps = sum v (2 n - d)
// (2^u), logs = sum v (c0 + ln m) (2^(u - 4)) over `positive` values, u = etop - 54.
__device__ __forceinline__ double node_entropy(double plus, long long steps, long long logs, int positive, int etop) {
  // in units of 2^(u - 3); the shifts of logs round down: half a unit per value on average
  const double x = fma(plus, (double)(etop + 2), 8.0 * (double)steps);
  const double l = 0.5 * ((double)logs + 0.5 * positive);
  return scaled(fma(x, LN2, fma(x, LN2_LOW, l)), etop - 57);
}

// Adds the NV values of v to the running mass, entropy, minimum and non-finite count; nnz(i) is
// the number of nonzero velocity components of value i.
template <typename V, int NV, typename Nnz>
__device__ __forceinline__ void add_values(const V (&v)[NV], Nnz nnz, const long long (&t)[LN_ENTRIES], double& mass,
                                           double& entropy, double& gmin, unsigned& bad) {
  using Man = typename std::conditional<sizeof(V) == 4, uint32_t, uint64_t>::type;
  if constexpr (sizeof(V) == 4) {
    // Almost every node has positive normal values within a factor 2^29 of one another: shifts
    // below 32, no signs, nothing to leave out (48 instructions per value instead of 89).
    constexpr uint32_t low_bits = 1u << 23;             // the smallest positive normal value
    uint32_t most = 0u, least = 0xffffffffu;
    float low = v[0];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const uint32_t b = __float_as_uint(v[i]) - low_bits;   // negative, zero, inf and NaN become large
      most = max(most, b);
      least = min(least, b);
      low = fminf(low, v[i]);
    }
    const int etop = (int)((most + low_bits) >> 23);    // biased
    if (most < 0x7f000000u && etop - (int)((least + low_bits) >> 23) <= 29) {
      long long plus = 0, steps = 0, logs = 0;          // units 2^(etop - 54), 2^(etop - 54), 2^(etop - 58)
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const uint32_t b = __float_as_uint(v[i]), man = (b & 0x7fffffu) | 0x800000u;
        const int d = etop - (int)(b >> 23);
        const uint32_t ahi = (man >> 1) >> d, alo = __funnelshift_r(man << 31, man >> 1, d);
        const long long a = (long long)((uint64_t)ahi << 32 | alo);   // man 2^31 >> d, exact
        plus += a;
        steps += a * (2 * nnz(i) - d);
        const long long q = v_ln_m(man, t);
        const uint32_t qlo = __funnelshift_r((uint32_t)q, (uint32_t)(q >> 32), d + 2);
        logs += (long long)((uint64_t)(uint32_t)((int)(q >> 32) >> (d + 2)) << 32 | qlo);
      }
      const double p = 8.0 * (double)plus;
      mass += scaled(p, etop - 127 - 57);
      entropy += node_entropy(p, steps, logs, NV, etop - 127);
      if (low < gmin) gmin = (double)low;
      return;
    }
  }
  V top = V(0), low = V(INFINITY);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const bool fin = value_finite(v[i]);
    bad += fin ? 0u : 1u;
    if (fin) {
      top = fmax(top, fabs(v[i]));
      low = fmin(low, v[i]);
    }
  }
  if (low < gmin) gmin = (double)low;
  Man man;
  int etop;
  bool neg;
  split_value(top, man, etop, neg);
  if (man == 0) return;
  // sums over the positive and the negative values (units 2^(etop - 57)), and over the positive
  // ones of v (2 n - d) (units 2^(etop - 54)) and v (c0 + ln m) (units 2^(etop - 58)); 27 values
  // of these units stay below 2^63
  long long plus = 0, minus = 0, steps = 0, logs = 0;
  int positive = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    int e;
    split_value(v[i], man, e, neg);
    if (man == 0 || !value_finite(v[i])) continue;
    const int d = min(etop - e, 63);
    const long long a = (long long)((unsigned long long)man << (sizeof(V) == 4 ? 34 : 5)) >> d;
    if (neg) {
      minus += a;
    } else {
      plus += a;
      steps += ((long long)man * (2 * nnz(i) - d) * (sizeof(V) == 4 ? (1ll << 31) : 4ll)) >> d;
      logs += v_ln_m(man, t) >> min(d + 2, 63);
      ++positive;
    }
  }
  const double p = (double)plus;
  mass += scaled(p - (double)minus, etop - 57);
  if (positive != 0) entropy += node_entropy(p, steps, logs, positive, etop);
}

#endif

}  // namespace elbm
