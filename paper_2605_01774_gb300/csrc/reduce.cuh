// Conservation diagnostics of a D3Q27 state: kernels shared by the handles (aux.cu) and by the
// allocation-free call (noalloc.cu).  Four partials per block (mass, entropy, min g, number of
// non-finite g), added in a fixed order by one block, so the result is deterministic.
#pragma once
#include "entropy.cuh"
#include "internal.h"
#include "pull.cuh"

namespace elbm {

// Most blocks of a reduction: 8 of 256 threads per SM of a GB300, each striding over the nodes.
constexpr int REDUCE_BLOCKS = 152 * 8;

inline int reduce_grid(size_t N) {
  const size_t want = (N + 255) / 256;
  return (int)(want < (size_t)REDUCE_BLOCKS ? want : (size_t)REDUCE_BLOCKS);
}

namespace {   // each translation unit has its own kernels and its own copy of the logarithm's table

// Adds the four sums over a block of 256 threads; thread 0 writes them to part[4 block ..].
__device__ __forceinline__ void block_partials(double m, double h, double gmin, double bad, double* __restrict__ part) {
  __shared__ double sm[4][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m += __shfl_xor_sync(0xffffffffu, m, o);
    h += __shfl_xor_sync(0xffffffffu, h, o);
    gmin = fmin(gmin, __shfl_xor_sync(0xffffffffu, gmin, o));
    bad += __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (lane == 0) {
    sm[0][wid] = m;
    sm[1][wid] = h;
    sm[2][wid] = gmin;
    sm[3][wid] = bad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0, c = 1.7976931348623157e308, d = 0;
    for (int w = 0; w < 8; ++w) {
      a += sm[0][w];
      b += sm[1][w];
      c = fmin(c, sm[2][w]);
      d += sm[3][w];
    }
    part[4 * blockIdx.x + 0] = a;
    part[4 * blockIdx.x + 1] = b;
    part[4 * blockIdx.x + 2] = c;
    part[4 * blockIdx.x + 3] = d;
  }
}

// PULL false: the stored populations are summed where they lie, plane by plane (streaming on a
// periodic lattice only permutes them); true: the pre-collision state is pulled node by node
// (Dirichlet faces, or a source half-step `half` * src * E_i in FP64).
// V: float for the FP32-arithmetic storages without a source, else double.
template <typename Elem, bool PULL, typename V>
__global__ void __launch_bounds__(256)
k_reduce_partials(Field<Elem> f, Grid G, const float* __restrict__ src, double half, double* __restrict__ part,
                  const PopConsts<typename Storage<Elem>::real> k) {
  using R = typename Storage<Elem>::real;
  __shared__ long long table[LN_ENTRIES];
  load_ln_table<3>(table);
  __syncthreads();
  double m = 0.0, h = 0.0, gmin = 1.7976931348623157e308;
  unsigned bad = 0;
  const int N = (int)G.N, stride = (int)(gridDim.x * blockDim.x);
  for (int n = (int)(blockIdx.x * blockDim.x + threadIdx.x); n < N; n += stride) {
    V v[Q];
    if constexpr (PULL) {
      const int x = n % G.nx, row = n / G.nx;
      R g[Q];
      pull_node<Elem, R>(g, f, G, x, row % G.ny, row / G.ny, k);
      const double r = src != nullptr ? half * (double)src[n] : 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = src != nullptr ? V((double)g[i] + r * (double)k.E[i]) : V(g[i]);
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = V(Storage<Elem>::load(f.pops, f.scale, N, i, n, k.E[i]));
    }
    add_values<V, Q>(v, [](int i) { return nnz_of(i); }, table, m, h, gmin, bad);
  }
  block_partials(m, h, gmin, (double)bad, part);
}

__global__ void __launch_bounds__(256) k_reduce_final(const double* __restrict__ part, int nblk,
                                                             double* __restrict__ out4) {
  __shared__ double sm[4][256];
  double a = 0, b = 0, c = 1.7976931348623157e308, d = 0;
  for (int i = threadIdx.x; i < nblk; i += 256) {
    a += part[4 * i];
    b += part[4 * i + 1];
    c = fmin(c, part[4 * i + 2]);
    d += part[4 * i + 3];
  }
  sm[0][threadIdx.x] = a;
  sm[1][threadIdx.x] = b;
  sm[2][threadIdx.x] = c;
  sm[3][threadIdx.x] = d;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      sm[0][threadIdx.x] += sm[0][threadIdx.x + s];
      sm[1][threadIdx.x] += sm[1][threadIdx.x + s];
      sm[2][threadIdx.x] = fmin(sm[2][threadIdx.x], sm[2][threadIdx.x + s]);
      sm[3][threadIdx.x] += sm[3][threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out4[0] = sm[0][0];
    out4[1] = sm[1][0];
    out4[2] = sm[2][0];
    out4[3] = sm[3][0];
  }
}

// part: 4 doubles per block of reduce_grid(N); out4: device.
template <typename Elem>
cudaError_t launch_reduce_t(const Field<Elem>& f, const Grid& G, const float* src, double half, double* part,
                            double* out4, const PopConsts<typename Storage<Elem>::real>& k, cudaStream_t s) {
  using R = typename Storage<Elem>::real;
  const int nblk = reduce_grid(G.N);
  if (src != nullptr) k_reduce_partials<Elem, true, double><<<nblk, 256, 0, s>>>(f, G, src, half, part, k);
  else if (G.dirichlet) k_reduce_partials<Elem, true, R><<<nblk, 256, 0, s>>>(f, G, nullptr, 0.0, part, k);
  else k_reduce_partials<Elem, false, R><<<nblk, 256, 0, s>>>(f, G, nullptr, 0.0, part, k);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_reduce_final<<<1, 256, 0, s>>>(part, nblk, out4);
  return cudaGetLastError();
}

}  // namespace

}  // namespace elbm
