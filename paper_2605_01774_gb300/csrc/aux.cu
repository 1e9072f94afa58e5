// State transfer, read-outs, conservation reductions and the tensor pre-pass.
#include "internal.h"
#include "launch.cuh"
#include "pull.cuh"
#include "reduce.cuh"

namespace elbm {

namespace {

// Threads per block of the state transfers, nodes dealt out in a row.
#ifndef ELBM_IO_THREADS
#define ELBM_IO_THREADS 64
#endif
constexpr int THREADS = ELBM_IO_THREADS;

// The transfers are launched like steps (launch.cuh); what the caller's kernels write is read with plain
// loads, which do not move over the wait.
template <typename T>
__device__ __forceinline__ double ld_in(const void* p, size_t idx) {
  return (double)static_cast<const T*>(p)[idx];
}

// E_i(u) at node d of a velocity field.
template <typename R>
__device__ __forceinline__ R shape_at(const float* u3, size_t N, int d, int i) {
  const R ux = u3[d], uy = u3[N + d], uz = u3[2 * N + d];
  const R cu = R(cx_of(i)) * ux + R(cy_of(i)) * uy + R(cz_of(i)) * uz;
  return R(w_of(i)) * (R(1) + R(3) * cu + R(4.5) * cu * cu - R(1.5) * (ux * ux + uy * uy + uz * uz));
}

// ---------------------------------------------------------------- write state
// Stored layout is post-collision: the next step pulls A_i(y) into node y + c_i
// and adds R E_i there.  To make the next step see the pre-collision state G
// (which already holds the trailing half source), store
//   A_i(y) = G_i(y + c_i) - (1/2) R(y + c_i) E_i         if y + c_i is a node,
//   A_i(y) = 2 W_i phi_w - (G_opp(i)(y) - (1/2) R(y) E_opp(i))   otherwise
// (anti-bounce-back inverted: the stored outgoing population of a wall node only
// feeds the entering opposite one).
template <typename Elem, typename Tin, int FROM_PHI>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)   // 128^3 FP64 with source 447 us, unbounded 530; 256^3 FP32 402, with 3 blocks 462
k_write(Elem* __restrict__ pops, float* __restrict__ scale, Grid G, const void* in, const float* src, const float* u3,
        unsigned long long* reset, const PopConsts<typename Storage<Elem>::real> k) {
  using R = typename Storage<Elem>::real;
  const unsigned m = blockIdx.x * (unsigned)THREADS + threadIdx.x, row = m / (unsigned)G.nx;
  const int x = (int)(m - row * (unsigned)G.nx), y = (int)(row % (unsigned)G.ny), z = (int)(row / (unsigned)G.ny);
  wait_for_previous();
  if (m == 0 && reset != nullptr) reset[0] = reset[3] = 0ull;
  if (z >= G.nz) return;
  const int n = (int)m;
  // All 27 destinations are loaded at once (wrapped, as if periodic), then the uniform cases, then
  // the faces: with the cases inside the loop every load waited for the one before it (256^3 FP32
  // 0.50 -> 0.40 ms, FP16 deviations 0.56 -> 0.39 ms).
  const int xs[3] = {x == 0 ? G.nx - 1 : x - 1, x, x + 1 == G.nx ? 0 : x + 1};
  const int ys[3] = {(y == 0 ? G.ny - 1 : y - 1) * G.nx, y * G.nx, (y + 1 == G.ny ? 0 : y + 1) * G.nx};
  const int nxy = G.nx * G.ny;
  const int zs[3] = {(z == 0 ? G.nz - 1 : z - 1) * nxy, z * nxy, (z + 1 == G.nz ? 0 : z + 1) * nxy};
  const auto dest = [&](int i) { return xs[cx_of(i) + 1] + ys[cy_of(i) + 1] + zs[cz_of(i) + 1]; };
  R a[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) a[i] = R(ld_in<Tin>(in, FROM_PHI ? (size_t)dest(i) : (size_t)i * G.N + dest(i)));
  if (FROM_PHI) {
    if (u3 == nullptr) {
#pragma unroll
      for (int i = 0; i < Q; ++i) a[i] = a[i] * k.E[i];
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) a[i] = a[i] * shape_at<R>(u3, G.N, dest(i), i);   // the velocity of that node
    }
  }
  if (src != nullptr) {
#pragma unroll
    for (int i = 0; i < Q; ++i) a[i] -= k.src_half * R(src[dest(i)]) * k.E[i];
  }
  if (G.dirichlet && (x == 0 || x == G.nx - 1)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const bool lo = cx_of(i) < 0 && x == 0, hi = cx_of(i) > 0 && x == G.nx - 1;
      if (lo || hi) {                  // leaves through x = -1/2 or x = Nx - 1/2
        const int o = opp_of(i);
        const R Eo = FROM_PHI && u3 != nullptr ? shape_at<R>(u3, G.N, n, o) : k.E[o];
        R v = FROM_PHI ? R(ld_in<Tin>(in, n)) * Eo : R(ld_in<Tin>(in, (size_t)o * G.N + n));
        if (src != nullptr) v -= k.src_half * R(src[n]) * k.E[o];
        a[i] = R(2.0 * w_of(i)) * (hi ? k.phi_hi : k.phi_lo) - v;
      }
    }
  }
  Storage<Elem>::store(pops, scale, G.N, n, a, k.Ek, R(NAN));
}

// ----------------------------------------------------------------- read state
template <typename Elem, typename Tout, int WHAT>
__global__ void __launch_bounds__(THREADS, 768 / THREADS)   // FP16 phi of 256^3: 281 us, with up to 2 or 4 blocks 367 and 304
k_read(Field<Elem> f, Grid G, Tout* __restrict__ out, Tout* __restrict__ qout,
       const typename Storage<Elem>::real* __restrict__ T6, const float* src, const float* u3,
       const PopConsts<typename Storage<Elem>::real> k) {
  using R = typename Storage<Elem>::real;
  const unsigned m = blockIdx.x * (unsigned)THREADS + threadIdx.x, row = m / (unsigned)G.nx;
  const int x = (int)(m - row * (unsigned)G.nx), y = (int)(row % (unsigned)G.ny), z = (int)(row / (unsigned)G.ny);
  wait_for_previous();
  if (z >= G.nz) return;
  const int n = (int)m;
  R g[Q];
  pull_node<Elem, R>(g, f, G, x, y, z, k);
  if (src != nullptr) {
    const R r = k.src_half * R(src[n]);
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] += r * k.E[i];
  }
  if (WHAT == 0) {
#pragma unroll
    for (int i = 0; i < Q; ++i) out[(size_t)i * G.N + n] = Tout(g[i]);
  } else {
    R phi, mx, my, mz;
    moments(g, phi, mx, my, mz);
    out[n] = Tout(phi);
    if (qout != nullptr) {
      // q = j - S j / 2 = T j / 2 with T = 2I - S (Eq. app-cube-lb-flux)
      R ux = k.ux, uy = k.uy, uz = k.uz;
      if (u3 != nullptr) {
        ux = u3[n];
        uy = u3[G.N + n];
        uz = u3[2 * G.N + n];
      }
      const R jx = mx - phi * ux, jy = my - phi * uy, jz = mz - phi * uz;
      const Sym6<R> T = load_T<R>(T6, G.N, n, k.T);
      R tx, ty, tz;
      sym_mul(T, jx, jy, jz, tx, ty, tz);
      qout[n] = Tout(R(0.5) * tx);
      qout[G.N + n] = Tout(R(0.5) * ty);
      qout[2 * G.N + n] = Tout(R(0.5) * tz);
    }
  }
}

// ---------------------------------------------------------------- tensor pre-pass
// T = 2I - S = 12 D (I + 6 D)^-1 per node, in FP64 (Eq. method-s-from-d with
// cs2 = 1/3, dt = 1), from Cartesian D or from (ln d_k, ZYZ angles).
__device__ void sym3_inverse(const double m[6], double inv[6], double& det) {
  const double a = m[0], b = m[1], c = m[2], d = m[3], e = m[4], f = m[5];
  const double A = d * f - e * e, B = c * e - b * f, C = b * e - c * d;
  det = a * A + b * B + c * C;
  const double id = 1.0 / det;
  inv[0] = A * id;
  inv[1] = B * id;
  inv[2] = C * id;
  inv[3] = (a * f - c * c) * id;
  inv[4] = (b * c - a * e) * id;
  inv[5] = (a * d - b * b) * id;
}

template <typename TT>
__global__ void k_tensor(const float* __restrict__ in, int is_params, TT* __restrict__ T6, size_t N,
                         unsigned long long* bad) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= N) return;
  double t6[6];
  if (is_params) {
    double t[3];
    for (int k = 0; k < 3; ++k) {
      const double dk = exp((double)in[k * N + n]);
      t[k] = 12.0 * dk / (1.0 + 6.0 * dk);
    }
    double sa, ca, sb, cb, sc, cc;
    sincos((double)in[3 * N + n], &sa, &ca);
    sincos((double)in[4 * N + n], &sb, &cb);
    sincos((double)in[5 * N + n], &sc, &cc);
    // R = Rz(a) Ry(b) Rz(c)
    const double R[3][3] = {{ca * cb * cc - sa * sc, -ca * cb * sc - sa * cc, ca * sb},
                            {sa * cb * cc + ca * sc, -sa * cb * sc + ca * cc, sa * sb},
                            {-sb * cc, sb * sc, cb}};
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int q = 0; q < 6; ++q) {
      double s = 0.0;
      for (int k = 0; k < 3; ++k) s += R[ia[q]][k] * t[k] * R[ib[q]][k];
      t6[q] = s;
    }
    if (!(isfinite(t[0]) && isfinite(t[1]) && isfinite(t[2]))) atomicAdd(bad, 1ull);
  } else {
    double D[6];
    for (int q = 0; q < 6; ++q) D[q] = in[q * N + n];
    // Sylvester criterion for SPD
    const double m1 = D[0], m2 = D[0] * D[3] - D[1] * D[1];
    const double det = D[0] * (D[3] * D[5] - D[4] * D[4]) - D[1] * (D[1] * D[5] - D[4] * D[2]) +
                       D[2] * (D[1] * D[4] - D[3] * D[2]);
    if (!(m1 > 0.0 && m2 > 0.0 && det > 0.0)) atomicAdd(bad, 1ull);
    double M[6] = {1.0 + 6.0 * D[0], 6.0 * D[1], 6.0 * D[2], 1.0 + 6.0 * D[3], 6.0 * D[4], 1.0 + 6.0 * D[5]};
    double Mi[6], dm;
    sym3_inverse(M, Mi, dm);
    // 12 D Mi (D and Mi commute, product symmetric)
    const double Dm[3][3] = {{D[0], D[1], D[2]}, {D[1], D[3], D[4]}, {D[2], D[4], D[5]}};
    const double Im[3][3] = {{Mi[0], Mi[1], Mi[2]}, {Mi[1], Mi[3], Mi[4]}, {Mi[2], Mi[4], Mi[5]}};
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int q = 0; q < 6; ++q) {
      double s = 0.0;
      for (int k = 0; k < 3; ++k) s += Dm[ia[q]][k] * Im[k][ib[q]];
      t6[q] = 12.0 * s;
    }
  }
  for (int q = 0; q < 6; ++q) T6[q * N + n] = (TT)t6[q];
}

template <typename Elem>
Field<Elem> field_of(const StateIO& S) {
  return Field<Elem>{static_cast<const Elem*>(S.pops), S.scale};
}

template <typename Elem>
const PopConsts<typename Storage<Elem>::real>& consts_of(const StateIO& S) {
  using R = typename Storage<Elem>::real;
  return *reinterpret_cast<const PopConsts<R>*>(std::is_same<R, double>::value ? (const void*)S.kd : (const void*)S.kf);
}

template <typename Elem>
cudaError_t write_t(const StateIO& S, const void* in, int in_f32, int from_phi, cudaStream_t s) {
  Grid G{S.nx, S.ny, S.nz, S.N, S.dirichlet};
  const dim3 b(THREADS), g((unsigned)((S.N + THREADS - 1) / THREADS));
  Elem* p = static_cast<Elem*>(S.pops);
  const auto& k = consts_of<Elem>(S);
  auto kernel = in_f32 ? (from_phi ? k_write<Elem, float, 1> : k_write<Elem, float, 0>)
                       : (from_phi ? k_write<Elem, double, 1> : k_write<Elem, double, 0>);
  return launch_next(kernel, g, b, 0, s, p, S.scale, G, in, S.src, S.u3, S.reset, k);
}

template <typename Elem>
cudaError_t read_t(const StateIO& S, void* out, void* q, int out_f32, int what, cudaStream_t s) {
  Grid G{S.nx, S.ny, S.nz, S.N, S.dirichlet};
  const dim3 b(THREADS), g((unsigned)((S.N + THREADS - 1) / THREADS));
  using R = typename Storage<Elem>::real;
  const auto& k = consts_of<Elem>(S);
  Field<Elem> f = field_of<Elem>(S);
  const R* T6 = static_cast<const R*>(S.T6);
  if (out_f32)
    return launch_next(what == 0 ? k_read<Elem, float, 0> : k_read<Elem, float, 1>, g, b, 0, s, f, G, (float*)out,
                       (float*)q, T6, S.src, S.u3, k);
  return launch_next(what == 0 ? k_read<Elem, double, 0> : k_read<Elem, double, 1>, g, b, 0, s, f, G, (double*)out,
                     (double*)q, T6, S.src, S.u3, k);
}

template <typename Elem>
cudaError_t reduce_t(const StateIO& S, double* scratch, double* out4, cudaStream_t s) {
  Grid G{S.nx, S.ny, S.nz, S.N, S.dirichlet};
  const auto& k = consts_of<Elem>(S);
  return launch_reduce_t<Elem>(field_of<Elem>(S), G, S.src, (double)k.src_half, scratch, out4, k, s);
}

}  // namespace

cudaError_t launch_write_state(const StateIO& S, const void* in, int in_f32, int from_phi, cudaStream_t s) {
  switch (S.prec) {
    case 0: return write_t<double>(S, in, in_f32, from_phi, s);
    case 1: return write_t<float>(S, in, in_f32, from_phi, s);
    case 2: return write_t<__half>(S, in, in_f32, from_phi, s);
    case 3: return write_t<__nv_bfloat16>(S, in, in_f32, from_phi, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_read_state(const StateIO& S, void* out, void* q, int out_f32, int what, cudaStream_t s) {
  switch (S.prec) {
    case 0: return read_t<double>(S, out, q, out_f32, what, s);
    case 1: return read_t<float>(S, out, q, out_f32, what, s);
    case 2: return read_t<__half>(S, out, q, out_f32, what, s);
    case 3: return read_t<__nv_bfloat16>(S, out, q, out_f32, what, s);
  }
  return cudaErrorInvalidValue;
}

size_t reduce_blocks(const StateIO& S) { return (size_t)reduce_grid(S.N); }

cudaError_t launch_reduce(const StateIO& S, double* scratch, double* out4, cudaStream_t s) {
  switch (S.prec) {
    case 0: return reduce_t<double>(S, scratch, out4, s);
    case 1: return reduce_t<float>(S, scratch, out4, s);
    case 2: return reduce_t<__half>(S, scratch, out4, s);
    case 3: return reduce_t<__nv_bfloat16>(S, scratch, out4, s);
  }
  return cudaErrorInvalidValue;
}

__global__ void k_velocity_check(const float* __restrict__ u3, size_t N, unsigned long long* bad) {
  const size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (n >= N) return;
  const double ux = u3[n], uy = u3[N + n], uz = u3[2 * N + n];
  bool ok = isfinite(ux) && isfinite(uy) && isfinite(uz);
  const double uu = ux * ux + uy * uy + uz * uz;
  for (int i = 0; i < Q && ok; ++i) {
    const double cu = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
    ok = 1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu > 0.0;
  }
  if (!ok) atomicAdd(bad, 1ull);
}

cudaError_t launch_velocity_check(const float* u3, size_t N, unsigned long long* bad, cudaStream_t s) {
  const int b = 256;
  k_velocity_check<<<(unsigned)((N + b - 1) / b), b, 0, s>>>(u3, N, bad);
  return cudaGetLastError();
}

cudaError_t launch_tensor_prepass(const float* in, int is_params, void* T6, int t6_f64, size_t N,
                                  unsigned long long* bad, cudaStream_t s) {
  const int b = 256;
  const size_t g = (N + b - 1) / b;
  if (t6_f64) k_tensor<double><<<(unsigned)g, b, 0, s>>>(in, is_params, static_cast<double*>(T6), N, bad);
  else k_tensor<float><<<(unsigned)g, b, 0, s>>>(in, is_params, static_cast<float*>(T6), N, bad);
  return cudaGetLastError();
}

}  // namespace elbm
