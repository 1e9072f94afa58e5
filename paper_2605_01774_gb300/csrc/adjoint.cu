// Hand-written adjoint of the collide-stream step for gradients of a
// concentration misfit with respect to per-node tensor parameters
// theta = (ln d1, ln d2, ln d3, a, b, c):  D = R diag(d) R^T, R = Rz(a) Ry(b) Rz(c),
// T = 2I - S = R diag(t) R^T with t_k = 12 d_k / (1 + 6 d_k)  (Eq. method-s-eigen).
//
// State variable: pre-collision populations G^n [27][N] (periodic lattice, uniform u).
// Forward step (push form of Eq. method-lbe): node y collides G^n(y) and writes
// G^{n+1}_i(y + c_i).  One step's vector-Jacobian product is then a gather:
//   Gbar^n(y) = J_C(G^n(y), T(y))^T [Gbar^{n+1}_i(y + c_i)]_i ,
//   Tbar(y)  += d/dT of the same,
// so every adjoint node update reads its 27 neighbours and writes only its own node: no
// atomics.  (With a pull forward step the transpose would scatter into 27 neighbours.)  The
// push stores are not scattered: for one population a warp writes 32 consecutive nodes shifted
// by c_x, i.e. two 128-byte segments, the same access shape as the pull kernel's loads.
// with the collision of collide.cuh (VEL = 1) differentiated by hand below.
// Misfit J = 1/2 sum_{t in obs} sum_x (phi_t(x) - phi*_t(x))^2, phi_t = sum_i G^t_i,
// enters the reverse sweep as Gbar^t_i(x) += phi_t(x) - phi*_t(x).
// The positivity fallback must stay inactive on gradient runs (its count is returned).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/elbm.h"
#include "../../include/elbm_adjoint.h"
#include "collide64.cuh"
#include "internal.h"
#include "launch.cuh"

using namespace elbm;

namespace {

// Threads per block of the step kernels.  FP64: 30 x 32 x 28 nodes are 105 blocks of 256 threads,
// fewer than SMs; blocks of 64 put the same warps on all of them.
template <typename R>
constexpr int STEP_THREADS = sizeof(R) == 8 ? 64 : 128;

// States of a run that are kept rather than recomputed, and the workspace that a handle keeps
// between calls (a larger one is given back at the end of the call), unless the caller sets another
// limit.  64^3 FP32 with 32 steps and
// checkpoints every 8 (3.1 ms a call) recomputed 28 of them, 14 us each, and got and returned 0.4 GB
// on each call.
constexpr size_t KEEP_BYTES = 4ull << 30;

struct AGrid {
  int nx, ny, nz;
  int N;
};

__device__ __forceinline__ void coords(const AGrid& G, int n, int& x, int& y, int& z) {
  x = n % G.nx;
  const int r = n / G.nx;
  y = r % G.ny;
  z = r / G.ny;
}

__device__ __forceinline__ int nb(const AGrid& G, int x, int y, int z, int dx, int dy, int dz) {
  x += dx;
  y += dy;
  z += dz;
  x = x < 0 ? x + G.nx : (x >= G.nx ? x - G.nx : x);
  y = y < 0 ? y + G.ny : (y >= G.ny ? y - G.ny : y);
  z = z < 0 ? z + G.nz : (z >= G.nz ? z - G.nz : z);
  return x + G.nx * (y + G.ny * z);
}

// sum_i c_i v_i, taken three populations (cz = -1, 0, 1 of one (cx, cy)) at a time.
template <typename R>
struct FirstMoment {
  R x = R(0), y = R(0), z = R(0);
  __device__ __forceinline__ void add(int p, R v0, R v1, R v2) {
    const int cx = p / 3 - 1, cy = p % 3 - 1;
    z += v2 - v0;
    const R s = v0 + v1 + v2;
    if (cy != 0) y = cy > 0 ? y + s : y - s;
    if (cx != 0) x = cx > 0 ? x + s : x - s;
  }
};

// c_i . v for all 27 velocities, as (cx vx + cy vy) + cz vz: the order in which den and its guard
// have always been rounded, so that the same nodes are stabilised.
template <typename R>
struct DotsXYZ {
  R d[Q];
  __device__ __forceinline__ DotsXYZ(R vx, R vy, R vz) {
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      const int cx = p / 3 - 1, cy = p % 3 - 1;
      const R x = cx == 0 ? R(0) : (cx > 0 ? vx : -vx);
      const R xy = cy == 0 ? x : (cx == 0 ? (cy > 0 ? vy : -vy) : (cy > 0 ? x + vy : x - vy));
      d[3 * p] = p == 4 ? -vz : xy - vz;
      d[3 * p + 1] = xy;
      d[3 * p + 2] = p == 4 ? vz : xy + vz;
    }
  }
};

// ---------------------------------------------------------------- parameters -> T
// What dL/dtheta needs besides T is kept: aux[12][N] holds sin and cos of a, b, c, then t_k, then
// dt_k / d ln d_k.
template <typename R>
__global__ void k_params_to_T(const R* __restrict__ th, R* __restrict__ T6, double* __restrict__ aux, int N) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const size_t S = N;
  double t[3];
  for (int k = 0; k < 3; ++k) {
    const double d = exp((double)th[k * N + n]), r = 1.0 / (1.0 + 6.0 * d);
    t[k] = 12.0 * d * r;
    aux[(6 + k) * S + n] = t[k];
    aux[(9 + k) * S + n] = t[k] * r;
  }
  double sa, ca, sb, cb, sc, cc;
  sincos((double)th[3 * N + n], &sa, &ca);
  sincos((double)th[4 * N + n], &sb, &cb);
  sincos((double)th[5 * N + n], &sc, &cc);
  const double v[6] = {sa, ca, sb, cb, sc, cc};
  for (int q = 0; q < 6; ++q) aux[q * S + n] = v[q];
  const double Rm[3][3] = {{ca * cb * cc - sa * sc, -ca * cb * sc - sa * cc, ca * sb},
                           {sa * cb * cc + ca * sc, -sa * cb * sc + ca * cc, sa * sb},
                           {-sb * cc, sb * sc, cb}};
  const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
  for (int q = 0; q < 6; ++q) {
    double s = 0.0;
    for (int k = 0; k < 3; ++k) s += Rm[ia[q]][k] * t[k] * Rm[ib[q]][k];
    T6[q * N + n] = (R)s;
  }
}

// dL/dtheta from the accumulated dL/dT (6 unique components, off-diagonals counted once).
// With G the symmetric full-matrix gradient and H = R^T G R (the principal frame):
// dL/dt_k = H_kk, and turning the frame by dw about its own axes changes T by R [dw]x diag(t) R^T
// plus its transpose, so dL/dw_x = 2 (t_y - t_z) H_yz and cyclic.  The angles turn it about
//   c: its z axis;  b: (sin c, cos c, 0);  a: the third row of R.
// FP64 issues at 1/64 of the FP32 rate, so the sines, exponentials and quotients are not repeated
// here (64^3 FP32: 221 -> 49 us).
template <typename R>
__global__ void k_Tbar_to_params(const double* __restrict__ aux, const double* __restrict__ Tbar,
                                 R* __restrict__ gth, int N) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const size_t S = N;
  const double sa = aux[n], ca = aux[S + n], sb = aux[2 * S + n], cb = aux[3 * S + n], sc = aux[4 * S + n],
               cc = aux[5 * S + n];
  const double t[3] = {aux[6 * S + n], aux[7 * S + n], aux[8 * S + n]};
  const double Gm[6] = {Tbar[n],           0.5 * Tbar[S + n],     0.5 * Tbar[2 * S + n],
                        Tbar[3 * S + n],   0.5 * Tbar[4 * S + n], Tbar[5 * S + n]};
  const double cbcc = cb * cc, cbsc = cb * sc;
  // columns of R
  const double q[3][3] = {{ca * cbcc - sa * sc, sa * cbcc + ca * sc, -sb * cc},
                          {-ca * cbsc - sa * cc, -sa * cbsc + ca * cc, sb * sc},
                          {ca * sb, sa * sb, cb}};
  double w[3][3];   // G times the columns
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    w[k][0] = Gm[0] * q[k][0] + Gm[1] * q[k][1] + Gm[2] * q[k][2];
    w[k][1] = Gm[1] * q[k][0] + Gm[3] * q[k][1] + Gm[4] * q[k][2];
    w[k][2] = Gm[2] * q[k][0] + Gm[4] * q[k][1] + Gm[5] * q[k][2];
  }
  const auto H = [&](int i, int k) { return q[i][0] * w[k][0] + q[i][1] * w[k][1] + q[i][2] * w[k][2]; };
#pragma unroll
  for (int k = 0; k < 3; ++k) gth[k * N + n] = (R)(H(k, k) * aux[(9 + k) * S + n]);
  const double wx = 2.0 * (t[1] - t[2]) * H(1, 2), wy = 2.0 * (t[2] - t[0]) * H(2, 0), wz = 2.0 * (t[0] - t[1]) * H(0, 1);
  gth[3 * N + n] = (R)(q[0][2] * wx + q[1][2] * wy + cb * wz);
  gth[4 * N + n] = (R)(sc * wx + cc * wy);
  gth[5 * N + n] = (R)wz;
}

// ---------------------------------------------------------------- forward (push)
// States are read with plain loads: the kernel may be resident while the one before it still writes
// them (launch.cuh).
template <typename R>
__global__ void __launch_bounds__(STEP_THREADS<R>)
k_adj_forward(const R* Gin, R* Gout, const R* __restrict__ T6, AGrid G, const PopConsts<R> k, unsigned long long* fb) {
  wait_for_previous();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  bool took = false;
  if (n < G.N) {
    R g[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = Gin[i * G.N + n];
    const Sym6<R> T{T6[n], T6[G.N + n], T6[2 * G.N + n], T6[3 * G.N + n], T6[4 * G.N + n], T6[5 * G.N + n]};
    R phi;
    took = collide_node<R, 1>(g, T, k, true, phi);
    int x, y, z;
    coords(G, n, x, y, z);
#pragma unroll
    for (int i = 0; i < Q; ++i) Gout[i * G.N + nb(G, x, y, z, cx_of(i), cy_of(i), cz_of(i))] = g[i];
  }
  const unsigned m = __ballot_sync(0xffffffffu, took);
  if (m && (threadIdx.x & 31) == 0) atomicAdd(fb, (unsigned long long)__popc(m));
}

// A node left to FP64 (collide64.cuh), out of line.
__device__ __noinline__ bool adj_node_f64(const double* Gin, double* Gout, const double* T6, const AGrid& G, int n,
                                          const PopConsts<double>& k) {
  double g[Q], phi;
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = Gin[i * G.N + n];
  const Sym6<double> T{T6[n], T6[G.N + n], T6[2 * G.N + n], T6[3 * G.N + n], T6[4 * G.N + n], T6[5 * G.N + n]};
  const bool took = collide_node<double, 1>(g, T, k, true, phi);
  int x, y, z;
  coords(G, n, x, y, z);
#pragma unroll
  for (int i = 0; i < Q; ++i) Gout[i * G.N + nb(G, x, y, z, cx_of(i), cy_of(i), cz_of(i))] = g[i];
  return took;
}

// The FP64 step with the fixed-point collision (fixed.cuh) that the lattice's own steps use:
// 30 x 32 x 28 nodes 34 -> 15.6 us a launch.
struct FixedStep {
  FixConsts fix;
  PopConsts<double> pop;
};
__global__ void __launch_bounds__(64, 6)
k_adj_forward_fixed(const double* Gin, double* Gout, const double* __restrict__ T6, const __grid_constant__ AGrid G,
                    const __grid_constant__ FixedStep c, unsigned long long* fb) {
  __shared__ int64_t kept[KEPT * 64];
  wait_for_previous();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const Lanes lanes{__ballot_sync(0xffffffffu, n < G.N), G.nx};
  bool took = false;
  if (n < G.N) {
    double g[Q], T[6];
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = Gin[i * G.N + n];
#pragma unroll
    for (int q = 0; q < 6; ++q) T[q] = T6[q * G.N + n];
    int x, y, z;
    coords(G, n, x, y, z);
    InShared<64> keep{kept + threadIdx.x};
    const auto out = [&](int i, double v) { Gout[i * G.N + nb(G, x, y, z, cx_of(i), cy_of(i), cz_of(i))] = v; };
    int etop;
    const Fixed f = collide_fixed<1>(g, T, 0.0, false, true, c.fix, keep, took, etop, out,
                                     [&](bool refuse) { return lanes.any(refuse); });
    __syncwarp(lanes.all);
    if (f == Fixed::SMALL_ALPHA) blend_given(keep, etop, c.fix, out, [&](int i) { return Gin[i * G.N + n]; });
    else if (f == Fixed::REFUSED) took = adj_node_f64(Gin, Gout, T6, G, n, c.pop);
  }
  const unsigned m = __ballot_sync(0xffffffffu, took);
  if (m && (threadIdx.x & 31) == 0) atomicAdd(fb, (unsigned long long)__popc(m));
}

// ---------------------------------------------------------------- one-step VJP
// Gbar_out(y) = J^T gathered adjoint; Tbar(y) = or += dL/dT (FP64 accumulators; `first` sets them);
// if target is given (an observation time), Gbar_out(y)_i += phi(y) - target(y).
// Bound by instruction issue (FP64: by its pipe), so c_i is never multiplied by: products c_i . v
// come from shared partial sums (DotsXYZ), sums over c_i v_i go by threes (FirstMoment), and dh_i is
// kept for the second pass: about 800 operations per node (were 1450; with the blocks of STEP_THREADS
// a launch for 64^3 FP32 takes 28 -> 22 us, FP64 30 x 32 x 28 94 -> 60 us).
template <typename R>
__global__ void __launch_bounds__(STEP_THREADS<R>, sizeof(R) == 4 ? 4 : 1)   // 64^3 FP32, whole call: 1.37, 1.21, 1.18 ms with 1, 3, 4
k_adj_vjp(const R* Gn, const R* Gbar_next, R* Gbar_out, const R* __restrict__ T6, double* Tbar,
          const R* __restrict__ target, AGrid G, const PopConsts<R> k, int first) {
  wait_for_previous();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= G.N) return;
  int x, y, z;
  coords(G, n, x, y, z);
  R g[Q], yb[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    g[i] = Gn[i * G.N + n];
    yb[i] = Gbar_next[i * G.N + nb(G, x, y, z, cx_of(i), cy_of(i), cz_of(i))];
  }
  const Sym6<R> T{T6[n], T6[G.N + n], T6[2 * G.N + n], T6[3 * G.N + n], T6[4 * G.N + n], T6[5 * G.N + n]};
  // ---- forward recomputation (collide.cuh, VEL = 1, fallback inactive)
  R phi, mx, my, mz;
  moments(g, phi, mx, my, mz);
  const R jx = mx - phi * k.ux, jy = my - phi * k.uy, jz = mz - phi * k.uz;
  R tx, ty, tz;
  sym_mul(T, jx, jy, jz, tx, ty, tz);
  const R ax = tx - jx, ay = ty - jy, az = tz - jz;
  // ---- reverse of g* = psi E - kappa g + 3 W c.b, psi = (1 + kappa) phi, b = a + kappa j
  R psib = R(0), kapb = R(0);
  FirstMoment<R> bb;
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    R w3[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int i = 3 * p + m;
      psib += yb[i] * k.E[i];
      kapb -= yb[i] * g[i];
      w3[m] = R(3.0 * w_of(i)) * yb[i];
    }
    bb.add(p, w3[0], w3[1], w3[2]);
  }
  kapb += psib * phi;
  kapb += bb.x * jx + bb.y * jy + bb.z * jz;
  R kappa = R(0);
  R phib = R(0);
  R abx = bb.x, aby = bb.y, abz = bb.z, jbx = R(0), jby = R(0), jbz = R(0);
  const R tiny = sizeof(R) == 4 ? R(1e-30) : R(1e-300);
  bool on = false;
  if (phi > tiny) {
    const R inv = R(1) / phi;
    R dh[Q];
    R num = R(0), den = R(0);
    const DotsXYZ<R> ca(ax * inv, ay * inv, az * inv);
    {
      const DotsXYZ<R> cj(jx * inv, jy * inv, jz * inv);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        dh[i] = g[i] * inv - k.E[i] - R(3.0 * w_of(i)) * cj.d[i];
        num += dh[i] * (k.K3[i] * ca.d[i] + k.L[i]);
        den += dh[i] * dh[i] * k.M[i];
      }
    }
    on = den > k.theta2;
    if (on) {
      kappa = num / den;
      const R numb = kapb / den;
      const R denb2 = R(-2) * numb * kappa;            // twice d/d den
      R invb = R(0);
      FirstMoment<R> apb, jpb;                         // a' = a inv, j' = j inv, inv = 1 / phi
#pragma unroll
      for (int p = 0; p < 9; ++p) {
        R cak[3], cjb[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const int i = 3 * p + m;
          const R t = k.K3[i] * ca.d[i] + k.L[i];
          const R dhb = numb * t + denb2 * (dh[i] * k.M[i]);
          cak[m] = dh[i] * k.K3[i];                    // d num / d (c_i . a'), times numb below
          cjb[m] = R(3.0 * w_of(i)) * dhb;             // -d / d (c_i . j')
          yb[i] = dhb * inv - kappa * yb[i];
          invb += dhb * g[i];
        }
        apb.add(p, cak[0], cak[1], cak[2]);
        jpb.add(p, cjb[0], cjb[1], cjb[2]);
      }
      const R apx = numb * apb.x, apy = numb * apb.y, apz = numb * apb.z;
      abx += apx * inv;
      aby += apy * inv;
      abz += apz * inv;
      invb += apx * ax + apy * ay + apz * az;
      jbx = kappa * bb.x - jpb.x * inv;
      jby = kappa * bb.y - jpb.y * inv;
      jbz = kappa * bb.z - jpb.z * inv;
      invb -= jpb.x * jx + jpb.y * jy + jpb.z * jz;
      phib = psib * (R(1) + kappa) - invb * inv * inv;
    }
  }
  if (!on) {                                           // kappa = 0
    phib = psib;
#pragma unroll
    for (int i = 0; i < Q; ++i) yb[i] = R(0);
  }
  // a = T j - j
  R Tax, Tay, Taz;
  sym_mul(T, abx, aby, abz, Tax, Tay, Taz);
  jbx += Tax - abx;
  jby += Tay - aby;
  jbz += Taz - abz;
  const R tb[6] = {abx * jx, abx * jy + aby * jx, abx * jz + abz * jx, aby * jy, aby * jz + abz * jy, abz * jz};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    // one writer per node: an addition without a returned value only keeps the sum off the thread's
    // path (64^3 FP32, 32 steps: 1.43 -> 1.21 ms a call)
    double* const acc = Tbar + q * (size_t)G.N + n;
    if (first) *acc = (double)tb[q];
    else atomicAdd(acc, (double)tb[q]);
  }
  // j = m - phi u ; m = sum c g ; phi = sum g
  phib -= k.ux * jbx + k.uy * jby + k.uz * jbz;
  if (target != nullptr) phib += phi - target[n];
  const DotsXYZ<R> cjb(jbx, jby, jbz);
#pragma unroll
  for (int i = 0; i < Q; ++i) Gbar_out[i * G.N + n] = yb[i] + (cjb.d[i] + phib);
}

// misfit contribution 1/2 sum (phi - target)^2 and phi-adjoint seed at the last step
template <typename R>
__global__ void __launch_bounds__(256)
k_adj_misfit(const R* __restrict__ Gs, const R* __restrict__ target, double* __restrict__ part, R* __restrict__ seed,
             int N) {
  __shared__ double sm[256];
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (n < N) {
    R phi = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) phi += Gs[i * N + n];
    const double d = (double)phi - (double)target[n];
    v = 0.5 * d * d;
    if (seed != nullptr) {
#pragma unroll
      for (int i = 0; i < Q; ++i) seed[i * N + n] = (R)d;
    }
  }
  sm[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

}  // namespace

struct elbm_adjoint_ctx {
  AGrid G{};
  int prec = 0;
  cudaStream_t stream = nullptr;
  double u[3] = {0, 0, 0};
  double theta = 1e-8;
  int K = 50;
  PopConsts<double> kd{};
  PopConsts<float> kf{};
  void* T6 = nullptr;              // [6][N] R
  double* Tbar = nullptr;          // [6][N]
  FixedStep fixed{};               // FP64 steps in fixed point
  double* aux = nullptr;           // [12][N] (k_params_to_T)
  void* states = nullptr;          // checkpoints and segment states
  size_t state_bytes = 0;
  size_t keep_bytes = KEEP_BYTES;
  void* gbar[2] = {nullptr, nullptr};
  double* part = nullptr;
  unsigned long long* fb = nullptr;
  std::string err;
};

namespace {

elbm_status afail(elbm_adjoint_ctx* h, elbm_status s, const std::string& m) {
  if (h) h->err = m;
  return s;
}
#define ACK(call, where)                                                                           \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return afail(h, e_ == cudaErrorMemoryAllocation ? ELBM_ERR_OOM : ELBM_ERR_CUDA,              \
                   std::string(where) + ": " + cudaGetErrorString(e_));                            \
  } while (0)

void consts_for(elbm_adjoint_ctx* h) {
  const double* u = h->u;
  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  PopConsts<double>& k = h->kd;
  for (int i = 0; i < Q; ++i) {
    const double cu = cx_of(i) * u[0] + cy_of(i) * u[1] + cz_of(i) * u[2];
    const double P = 1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu;
    k.E[i] = w_of(i) * P;
    k.K3[i] = 3.0 * (1.0 / P - 1.0);
    k.L[i] = std::log(P) - 3.0 * cu + 1.5 * uu;
    k.M[i] = 1.0 / (w_of(i) * P);
  }
  k.ux = u[0];
  k.uy = u[1];
  k.uz = u[2];
  k.theta2 = h->theta * h->theta;
  k.eps = 0.0;
  PopConsts<float>& f = h->kf;
  for (int i = 0; i < Q; ++i) {
    f.E[i] = (float)k.E[i];
    f.K3[i] = (float)k.K3[i];
    f.L[i] = (float)k.L[i];
    f.M[i] = (float)k.M[i];
  }
  f.ux = (float)u[0];
  f.uy = (float)u[1];
  f.uz = (float)u[2];
  f.theta2 = (float)k.theta2;
  f.eps = 0.f;
  h->fixed.fix = fix_consts(h->kd);
  h->fixed.pop = h->kd;
}

template <typename R>
const PopConsts<R>& kc(elbm_adjoint_ctx* h);
template <>
const PopConsts<double>& kc<double>(elbm_adjoint_ctx* h) {
  return h->kd;
}
template <>
const PopConsts<float>& kc<float>(elbm_adjoint_ctx* h) {
  return h->kf;
}

int blocks(int N) { return (N + 255) / 256; }

template <typename R>
__global__ void k_adj_init(const R* __restrict__ phi0, R* __restrict__ Gs, int N, const PopConsts<R> k) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const R p = phi0[n];
#pragma unroll
  for (int i = 0; i < Q; ++i) Gs[i * N + n] = p * k.E[i];
}

int step_blocks(int N, int threads) { return (N + threads - 1) / threads; }

// One forward step (fallback nodes counted in *fb).
template <typename R>
cudaError_t forward(elbm_adjoint_ctx* h, const R* in, R* out, unsigned long long* fb) {
  const R* T6 = static_cast<const R*>(h->T6);
  if constexpr (sizeof(R) == 8) {
    if (h->fixed.fix.ok)
      return launch_next(k_adj_forward_fixed, dim3(step_blocks(h->G.N, 64)), dim3(64), 0, h->stream, in, out, T6, h->G,
                         h->fixed, fb);
  }
  constexpr int B = STEP_THREADS<R>;
  return launch_next(k_adj_forward<R>, dim3(step_blocks(h->G.N, B)), dim3(B), 0, h->stream, in, out, T6, h->G, kc<R>(h), fb);
}

template <typename R>
cudaError_t vjp(elbm_adjoint_ctx* h, const R* state, const R* gbar_next, R* gbar, const R* target, bool first) {
  constexpr int B = STEP_THREADS<R>;
  return launch_next(k_adj_vjp<R>, dim3(step_blocks(h->G.N, B)), dim3(B), 0, h->stream, state, gbar_next, gbar,
                     static_cast<const R*>(h->T6), h->Tbar, target, h->G, kc<R>(h), first ? 1 : 0);
}

// Whether all states of a run may be kept: within the handle's limit, and within half of the memory
// that is free for them.
bool may_keep(const elbm_adjoint_ctx* h, size_t bytes) {
  if (bytes > h->keep_bytes) return false;
  if (bytes <= h->state_bytes) return true;
  size_t free = 0, total = 0;
  return cudaMemGetInfo(&free, &total) == cudaSuccess && bytes <= (free + h->state_bytes) / 2;
}

// Room for `bytes` of states in the handle's workspace.
cudaError_t reserve(elbm_adjoint_ctx* h, size_t bytes) {
  if (bytes <= h->state_bytes) return cudaSuccess;
  cudaStreamSynchronize(h->stream);
  cudaFree(h->states);
  h->states = nullptr;
  h->state_bytes = 0;
  const cudaError_t e = cudaMalloc(&h->states, bytes);
  if (e == cudaSuccess) h->state_bytes = bytes;
  else cudaGetLastError();
  return e;
}

template <typename R>
elbm_status run_steps(elbm_adjoint_ctx* h, const R* theta, const R* phi0, int64_t nsteps, int nobs, const int64_t* obs,
                      const R* targets, double* J, R* grad, int64_t* nfb) {
  const int N = h->G.N;
  const size_t S = 27ull * N, sb = S * sizeof(R);
  cudaStream_t s = h->stream;
  // Segments of K steps.  A forward run alone alternates between two states.  With a gradient, every
  // state of the run is kept where that is allowed (one segment); else checkpoints every h->K steps,
  // and the states of one segment at a time.
  int64_t K = nsteps, last = 0, t_last = 0;     // last segment, its first step
  size_t ncheck = 1, nseg = 2;
  const auto plan = [&](int64_t every) {
    K = std::min<int64_t>(every, nsteps);
    last = (nsteps - 1) / K;
    t_last = last * K;
    ncheck = (size_t)last + 1;
    nseg = (size_t)K + 1;
  };
  if (grad != nullptr)
    plan(nsteps > h->K && (size_t)(nsteps + 2) <= h->keep_bytes / sb && may_keep(h, (size_t)(nsteps + 2) * sb) ? nsteps : h->K);
  cudaError_t e = reserve(h, (ncheck + nseg) * sb);
  if (e == cudaErrorMemoryAllocation && grad != nullptr && K > h->K) {
    plan(h->K);
    e = reserve(h, (ncheck + nseg) * sb);
  }
  ACK(e, "state buffer");
  R* const ck = static_cast<R*>(h->states);
  R* const seg = ck + S * ncheck;
  k_params_to_T<R><<<blocks(N), 256, 0, s>>>(theta, static_cast<R*>(h->T6), h->aux, N);
  ACK(cudaGetLastError(), "params");
  ACK(cudaMemsetAsync(h->fb, 0, 2 * sizeof(unsigned long long), s), "memset");
  ACK(cudaMemsetAsync(h->part, 0, sizeof(double) * blocks(N) * nobs, s), "memset");
  auto obs_index = [&](int64_t t) {
    for (int o = 0; o < nobs; ++o)
      if (obs[o] == t) return o;
    return -1;
  };
  R* gin = static_cast<R*>(h->gbar[0]);    // Gbar^{t+1}
  R* gout = static_cast<R*>(h->gbar[1]);   // Gbar^t
  // forward sweep: checkpoints every K steps, all states of the last segment, misfit at the
  // observation steps (at the last step it is also the seed Gbar^T_i = phi_T - target)
  k_adj_init<R><<<blocks(N), 256, 0, s>>>(phi0, ck, N, kc<R>(h));
  ACK(cudaGetLastError(), "init");
  const R* cur = ck;
  for (int64_t t = 0; t < nsteps; ++t) {
    R* dst;
    if (grad != nullptr && t >= t_last) dst = seg + S * (t + 1 - t_last);
    else if (grad != nullptr && (t + 1) % K == 0) dst = ck + S * ((t + 1) / K);
    else dst = cur == seg ? seg + S : seg;
    ACK(forward<R>(h, cur, dst, h->fb), "forward");
    cur = dst;
    const int o = obs_index(t + 1);
    if (o >= 0) {
      k_adj_misfit<R><<<blocks(N), 256, 0, s>>>(cur, targets + (size_t)o * N, h->part + (size_t)o * blocks(N),
                                               grad != nullptr && t + 1 == nsteps ? gin : nullptr, N);
      ACK(cudaGetLastError(), "misfit");
    }
  }
  if (grad != nullptr) {
    // reverse sweep, segment by segment from the end
    if (obs_index(nsteps) < 0) ACK(cudaMemsetAsync(gin, 0, sb, s), "memset");
    for (int64_t sgm = last; sgm >= 0; --sgm) {
      const int64_t t0 = sgm * K;
      const int64_t t1 = std::min<int64_t>(nsteps, t0 + K);
      const auto state = [&](int64_t t) { return t == t0 ? ck + S * sgm : seg + S * (t - t0); };
      if (sgm != last)
        for (int64_t t = t0; t < t1 - 1; ++t) ACK(forward<R>(h, state(t), state(t + 1), h->fb + 1), "recompute");
      for (int64_t t = t1 - 1; t >= t0; --t) {
        const int o = obs_index(t);
        const R* tgt = (o >= 0 && t > 0) ? targets + (size_t)o * N : nullptr;
        ACK(vjp<R>(h, state(t), gin, gout, tgt, t == nsteps - 1), "vjp");
        std::swap(gin, gout);
      }
    }
    k_Tbar_to_params<R><<<blocks(N), 256, 0, s>>>(h->aux, h->Tbar, grad, N);
    ACK(cudaGetLastError(), "chain rule");
  }
  std::vector<double> part((size_t)blocks(N) * nobs);
  ACK(cudaMemcpyAsync(part.data(), h->part, part.size() * sizeof(double), cudaMemcpyDeviceToHost, s), "memcpy");
  unsigned long long fb = 0;
  ACK(cudaMemcpyAsync(&fb, h->fb, sizeof(fb), cudaMemcpyDeviceToHost, s), "memcpy");
  ACK(cudaStreamSynchronize(s), "sync");
  double Jv = 0.0;
  for (double v : part) Jv += v;
  if (J) *J = Jv;
  if (nfb) *nfb = (int64_t)fb;
  return ELBM_OK;
}

void release_states(elbm_adjoint_ctx* h) {
  cudaStreamSynchronize(h->stream);
  cudaFree(h->states);
  h->states = nullptr;
  h->state_bytes = 0;
}

template <typename R>
elbm_status run_t(elbm_adjoint_ctx* h, const R* theta, const R* phi0, int64_t nsteps, int nobs, const int64_t* obs,
                  const R* targets, double* J, R* grad, int64_t* nfb) {
  const elbm_status st = run_steps<R>(h, theta, phi0, nsteps, nobs, obs, targets, J, grad, nfb);
  if (h->state_bytes > h->keep_bytes) release_states(h);
  return st;
}

}  // namespace

extern "C" {

elbm_status elbm_adjoint_create(const int64_t dims[3], elbm_precision prec, void* cuda_stream,
                                elbm_adjoint_handle* out) {
  if (!dims || !out) return ELBM_ERR_ARG;
  *out = nullptr;
  if (prec != ELBM_F64 && prec != ELBM_F32) return ELBM_ERR_UNSUPPORTED;
  for (int a = 0; a < 3; ++a)
    if (dims[a] < 1 || dims[a] > 4096) return ELBM_ERR_ARG;
  const double N = (double)dims[0] * dims[1] * dims[2];
  if (27.0 * N >= 2147483647.0) return ELBM_ERR_ARG;
  elbm_adjoint_ctx* h = new elbm_adjoint_ctx();
  h->G = AGrid{(int)dims[0], (int)dims[1], (int)dims[2], (int)N};
  h->prec = (int)prec;
  h->stream = static_cast<cudaStream_t>(cuda_stream);
  const size_t rs = prec == ELBM_F64 ? 8 : 4;
  cudaError_t e = cudaMalloc(&h->T6, 6 * (size_t)N * rs);
  if (e == cudaSuccess) e = cudaMalloc((void**)&h->Tbar, 6 * (size_t)N * sizeof(double));
  for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMalloc(&h->gbar[b], 27 * (size_t)N * rs);
  if (e == cudaSuccess) e = cudaMalloc((void**)&h->aux, 12 * (size_t)N * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc((void**)&h->fb, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMalloc((void**)&h->part, sizeof(double) * blocks((int)N) * 16);
  if (e != cudaSuccess) {
    elbm_adjoint_destroy(h);
    return e == cudaErrorMemoryAllocation ? ELBM_ERR_OOM : ELBM_ERR_CUDA;
  }
  consts_for(h);
  *out = h;
  return ELBM_OK;
}

void elbm_adjoint_destroy(elbm_adjoint_handle h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  cudaFree(h->T6);
  cudaFree(h->Tbar);
  cudaFree(h->gbar[0]);
  cudaFree(h->gbar[1]);
  cudaFree(h->aux);
  cudaFree(h->states);
  cudaFree(h->fb);
  cudaFree(h->part);
  delete h;
}

const char* elbm_adjoint_last_error(elbm_adjoint_handle h) { return h ? h->err.c_str() : "null handle"; }

elbm_status elbm_adjoint_configure(elbm_adjoint_handle h, const double u[3], double theta, int32_t checkpoint_every) {
  if (!h || !u || !(theta >= 0.0) || checkpoint_every < 1) return afail(h, ELBM_ERR_ARG, "bad argument");
  if (elbm_check_velocity(u) != ELBM_OK) return afail(h, ELBM_ERR_MACH, "velocity gives a non-positive P_i(u)");
  std::memcpy(h->u, u, sizeof(h->u));
  h->theta = theta;
  h->K = checkpoint_every;
  consts_for(h);
  return ELBM_OK;
}

elbm_status elbm_adjoint_set_workspace(elbm_adjoint_handle h, size_t bytes) {
  if (!h) return ELBM_ERR_ARG;
  h->keep_bytes = bytes;
  if (h->state_bytes > bytes) release_states(h);
  return ELBM_OK;
}

elbm_status elbm_adjoint_misfit(elbm_adjoint_handle h, const void* theta6, const void* phi0, int64_t nsteps,
                                int32_t nobs, const int64_t* obs_steps, const void* targets, double* J, void* grad6,
                                int64_t* n_fallback) {
  if (!h || !theta6 || !phi0 || nsteps < 1 || nobs < 1 || nobs > 16 || !obs_steps || !targets)
    return afail(h, ELBM_ERR_ARG, "bad argument");
  for (int o = 0; o < nobs; ++o)
    if (obs_steps[o] < 1 || obs_steps[o] > nsteps) return afail(h, ELBM_ERR_ARG, "observation step out of range");
  if (h->prec == ELBM_F64)
    return run_t<double>(h, (const double*)theta6, (const double*)phi0, nsteps, nobs, obs_steps,
                         (const double*)targets, J, (double*)grad6, n_fallback);
  return run_t<float>(h, (const float*)theta6, (const float*)phi0, nsteps, nobs, obs_steps, (const float*)targets, J,
                      (float*)grad6, n_fallback);
}

}  // extern "C"

template <typename R>
static elbm_status step_t(elbm_adjoint_ctx* h, const R* theta, const R* g, const R* gbar_next, R* g_next, R* gbar,
                          R* grad) {
  const int N = h->G.N;
  cudaStream_t s = h->stream;
  k_params_to_T<R><<<blocks(N), 256, 0, s>>>(theta, static_cast<R*>(h->T6), h->aux, N);
  ACK(cudaGetLastError(), "params");
  // (also keeps the step kernels, which may start before the kernel in front of them ends, from
  // meeting an unfinished T6)
  ACK(cudaMemsetAsync(h->fb, 0, 2 * sizeof(unsigned long long), s), "memset");
  if (g_next) ACK(forward<R>(h, g, g_next, h->fb), "forward");
  if (gbar) {
    ACK(vjp<R>(h, g, gbar_next, gbar, nullptr, true), "vjp");
    if (grad) {
      k_Tbar_to_params<R><<<blocks(N), 256, 0, s>>>(h->aux, h->Tbar, grad, N);
      ACK(cudaGetLastError(), "chain rule");
    }
  }
  ACK(cudaStreamSynchronize(s), "sync");
  return ELBM_OK;
}

extern "C" {

elbm_status elbm_adjoint_step(elbm_adjoint_handle h, const void* theta6, const void* g, const void* gbar_next,
                              void* g_next, void* gbar, void* grad6) {
  if (!h || !theta6 || !g || (gbar && !gbar_next)) return afail(h, ELBM_ERR_ARG, "bad argument");
  if (h->prec == ELBM_F64)
    return step_t<double>(h, (const double*)theta6, (const double*)g, (const double*)gbar_next, (double*)g_next,
                          (double*)gbar, (double*)grad6);
  return step_t<float>(h, (const float*)theta6, (const float*)g, (const float*)gbar_next, (float*)g_next,
                       (float*)gbar, (float*)grad6);
}

}  // extern "C"
