// The collision of a pulled node with its source term, as every step kernel calls it: FP64 nodes of
// a uniform velocity go through the fixed-point collision (fixed.cuh), all others through
// collide_node.
#pragma once
#include "fixed.cuh"
#include "pull.cuh"

namespace elbm {

// How a step kernel collides: in floating point with the closed-form stabilizer or with its exact
// root, or (FP64) in fixed point.
enum : int { CLOSED = 0, ROOT = 1, FIXED = 2 };

// What a step kernel is given besides PopConsts: the fixed-point constants where it uses them.
template <int MODE>
struct StepConsts {};
template <>
struct StepConsts<FIXED> {
  FixConsts fix;
  PopConsts<double> pop;   // for the functions out of line, which take its address
};

template <int MODE, typename Launch>
inline StepConsts<MODE> step_consts(const Launch& L) {
  StepConsts<MODE> c{};
  if constexpr (MODE == FIXED) {
    c.fix = *L.fix;
    c.pop = *L.kd;
  }
  return c;
}

// Pull, FP64 collision and store of a node that is left to FP64.
//
// One node that fixed point cannot hold keeps its warp's FP64 pipe busy for the whole FP64 collision,
// whichever lanes take part, so the warp's other nodes go with it (Lanes) rather than through the
// integer collision as well.  (Such nodes are rare near equilibrium, but steep tails consist of them: of the
// 256^3 plume of width 8 they are 20 % at step 2 and 62 % at step 24.)  Steps of a 96 x 80 x 72 plume
// of width 2 took 0.68, 0.86 and 1.01 ms (20 steps each) with both collisions in such warps, 0.63, 0.70
// and 0.76 with one, 0.66, 0.73 and 0.77 with FP64 arithmetic alone; of width 4 0.69 to 0.84, 0.61 to
// 0.70, 0.68 to 0.74; of 128^3 with width 8 0.84 to 1.97 (first 20 to 120 steps), 0.79 to 1.75, 1.96 to
// 2.29; of 256^3 14.6 to 21.1 (first 10 to 80), 13.1 to 17.7, 17.8 to 20.1.
template <int VEL>
__device__ __forceinline__ bool step_node_f64(const Field<double>& in, const Grid& G, int n, const Sym6<double>& T, double r,
                                           bool has_src, const PopConsts<double>& k, bool fallback, double* out) {
  double g[Q], phi;
  const int row = n / G.nx;
  pull_node<double, double>(g, in, G, n - row * G.nx, row % G.ny, row / G.ny, k);
  if (has_src) {
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] += r * k.E[i];
  }
  const bool took = collide_node<double, VEL>(g, T, k, fallback, phi);
  Storage<double>::store(out, nullptr, (int)G.N, n, g, k.Ek, phi);
  return took;
}

// The same out of line, for u != 0: inline it takes 2 % longer where most nodes come here (96 x 80 x 72
// plume 2 wide 0.70 -> 0.72 ms a step).  At u = 0 inline is faster (0.418 -> 0.409), also for the other
// nodes (8 wide 0.087 -> 0.085 ms, with a floor 67.6 -> 64.9 us).
template <int VEL>
__device__ __noinline__ bool step_node_f64_out(const Field<double>& in, const Grid& G, int n, const Sym6<double>& T,
                                               double r, bool has_src, const PopConsts<double>& k, bool fallback,
                                               double* out) {
  return step_node_f64<VEL>(in, G, n, T, r, has_src, k, fallback, out);
}

// The lanes of a warp that have a node, and those of them whose nodes are left to FP64 together: 32
// neighbours in the order of the nodes, or 16 or 8 where rows are whole multiples of no more.  So the
// groups are the same nodes in every step kernel (the staged ones begin a warp at each row, and need
// rows of a multiple of 8), whose results stay bit-equal.
struct Lanes {
  unsigned all;
  int nx;
  // Whether a node of the group is refused; all of `all` call it.
  __device__ __forceinline__ bool any(bool refuse) const {
    const unsigned m = __ballot_sync(all, refuse);
    if (m == 0u) return false;
    const unsigned size = nx % 8 != 0 || nx % 32 == 0 ? 32u : (nx % 16 == 0 ? 16u : 8u);
    return (m & ((0xffffffffu >> (32u - size)) << (threadIdx.x & 31u & ~(size - 1u)))) != 0u;
  }
};

// Population i pulled into node n once more, with its source (src null: none); i not known at compile
// time.
static __device__ __noinline__ double pull_one(const Field<double>& in, const Grid& G, int n, int i, const float* src,
                                               const PopConsts<double>& k) {
  const int row = n / G.nx, x = n - row * G.nx, y = row % G.ny, z = row / G.ny;
  const int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
  double g;
  if (G.dirichlet && ((cx == 1 && x == 0) || (cx == -1 && x == G.nx - 1))) {
    g = 2.0 * w_of(i) * (x == 0 && cx == 1 ? k.phi_lo : k.phi_hi) - in.pops[(size_t)opp_of(i) * G.N + n];
  } else {
    const int sx = x < cx ? G.nx - 1 : (x - cx == G.nx ? 0 : x - cx);
    const int sy = y < cy ? G.ny - 1 : (y - cy == G.ny ? 0 : y - cy);
    const int sz = z < cz ? G.nz - 1 : (z - cz == G.nz ? 0 : z - cz);
    g = in.pops[(size_t)i * G.N + (size_t)(sx + G.nx * (sy + G.ny * sz))];
  }
  return src != nullptr ? g + k.src_step * (double)src[n] * k.E[i] : g;
}

// Collides g_i + r E_i (src, the source field, null: r is 0), g the populations pulled into node n of the lattice G
// from `in`, with the node's T where has_T, else the uniform one, and stores the result in `pout`,
// `sout`.  Returns whether the positivity fallback was taken; proj as Storage::store returns it.
// keep: where fixed point keeps the node's integers.  All of `lanes` call this together.
template <typename R, int VEL, int MODE, typename Elem, typename Keep>
__device__ __forceinline__ bool collide_and_store(R (&g)[Q], const Field<Elem>& in, Elem* __restrict__ pout,
                                                  float* __restrict__ sout, const Grid& G, int n, const Sym6<R>& T,
                                                  bool has_T, R r, const float* src, const PopConsts<R>& k,
                                                  const StepConsts<MODE>& c, bool fallback, const Lanes& lanes, Keep& keep,
                                                  bool& proj, const R* un = nullptr) {
  if constexpr (MODE == FIXED) {
    bool took;
    int etop;
    const double t6[6] = {T.xx, T.xy, T.xz, T.yy, T.yz, T.zz};
    proj = false;
    const auto out = [&](int i, double v) { pout[(size_t)i * G.N + n] = v; };
    const Fixed f = collide_fixed<VEL>(g, has_T ? t6 : nullptr, r, src != nullptr, fallback, c.fix, keep, took, etop, out,
                                       [&](bool refuse) { return lanes.any(refuse); });
    __syncwarp(lanes.all);
    if (f == Fixed::SMALL_ALPHA)
      blend_given(keep, etop, c.fix, out, [&](int i) { return pull_one(in, G, n, i, src, c.pop); });
    else if (f == Fixed::REFUSED)
      took = VEL == 0 ? step_node_f64<0>(in, G, n, T, r, src != nullptr, k, fallback, pout)
                      : step_node_f64_out<1>(in, G, n, T, r, src != nullptr, c.pop, fallback, pout);
    return took;
  } else {
    if (src != nullptr) {
#pragma unroll
      for (int i = 0; i < Q; ++i) g[i] += r * k.E[i];
    }
    R phi;
    const bool took = collide_node<R, VEL, MODE == ROOT>(g, T, k, fallback, phi, un);
    proj = Storage<Elem>::store(pout, sout, (int)G.N, n, g, k.Ek, phi, k.exact_mass != 0);
    return took;
  }
}

// Nothing to keep (floating-point collisions).
struct KeepNone {};
template <int MODE>
using KeepLocal = typename std::conditional<MODE == FIXED, InLocal, KeepNone>::type;

}  // namespace elbm
