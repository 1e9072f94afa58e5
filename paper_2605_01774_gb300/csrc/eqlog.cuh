// Per-population tables of a node's own velocity in FP32 (per-node velocity fields), shared by
// the D3Q27 and D2Q9 kernels.
//
// With a = 3 c.u - 1.5 u.u and b = 4.5 (c.u)^2, the equilibrium polynomial is P = 1 + t,
// t = a + b (Section 2.2), and the stabilizer needs
//     K3 = 3 (1/P - 1) = -3 t / P,   L = ln P - a,   M = 1 / (W P).
// L is O(u^3) while ln P and a are O(u): evaluated as written, the rounding of ln P (about
// 1e-8 absolute) is most of L.  With ln P = 2 artanh(s), s = t / (2 + t), and 2 s = t - t s,
//     L = b - t s + 2 s^3 (1/3 + s^2/5 + s^4/7 + ...),
// where the O(u) terms have cancelled analytically and the remaining O(u^2) ones (b, t s) are
// about ten times smaller than ln P.  The odd series of artanh is summed to s^15, which for
// |s| <= 0.3 (P in [0.54, 1.86]) leaves a truncation below 3e-9 of its leading term; outside
// that range L falls back to logf(P) - a.
//
// Choosing per population makes 27 branches that the tables' long chains (two quotients, the
// series) cannot be moved across, and a D3Q27 step waits for each chain in turn.  series_range tells
// once per node whether all populations lie inside: t is monotonic in c.u for |c.u| < 1/3, so its
// extremes over the velocity set are those of c.u = +-(|ux| + |uy| + |uz|), both attained.  With the
// tables computed where they are used (collide.cuh) 16 steps of 160 x 144 x 128 nodes and their
// read-outs take 4.13 -> 2.68 ms, of 40 x 50 x 37 nodes (10 steps) 171 -> 119 us.  D2Q9 (nine chains,
// 75 % of its issue slots used) gained nothing and chooses per population.
#pragma once

namespace elbm {

// m = |ux| + |uy| (+ |uz|), uu = u.u: whether |s| <= 0.3 for every population (with a margin above
// the rounding of t).
__device__ __forceinline__ bool series_range(float m, float uu) {
  const float even = 4.5f * m * m - 1.5f * uu;
  return m < 0.33f && even - 3.0f * m > -0.4614f && even + 3.0f * m < 0.857f;
}

// SERIES: every population is known to lie in the series' range.
// Every operation is an explicit intrinsic, so that each kernel that inlines this gets the
// same roundings (no contraction of b into t decided per call site).
template <bool SERIES>
__device__ __forceinline__ void eq_tables_f32(float a, float b, float w, float& E, float& K3, float& L, float& M) {
  const float t = __fadd_rn(a, b);
  const float P = __fadd_rn(1.0f, t);
  const float rP = __fdividef(1.0f, P);
  E = __fmul_rn(w, P);
  K3 = __fmul_rn(__fmul_rn(-3.0f, t), rP);
  M = __fmul_rn(rP, 1.0f / w);
  const float s = __fdividef(t, __fadd_rn(2.0f, t));
  if (SERIES || fabsf(s) <= 0.3f) {
    const float q = __fmul_rn(s, s);
    float p = 1.0f / 15.0f;
    p = fmaf(p, q, 1.0f / 13.0f);
    p = fmaf(p, q, 1.0f / 11.0f);
    p = fmaf(p, q, 1.0f / 9.0f);
    p = fmaf(p, q, 1.0f / 7.0f);
    p = fmaf(p, q, 1.0f / 5.0f);
    p = fmaf(p, q, 1.0f / 3.0f);
    L = fmaf(__fmul_rn(__fmul_rn(2.0f, s), q), p, fmaf(-t, s, b));
  } else {
    L = __fsub_rn(logf(P), a);
  }
}

}  // namespace elbm
