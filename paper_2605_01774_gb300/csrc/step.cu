// Fused collide-stream kernel: one thread per node pulls its 27 populations,
// collides them in registers (collide.cuh) and writes the 27 post-collision
// values to its own node of the other buffer (coalesced writes, A/B buffers).
#include "collide64.cuh"
#include "internal.h"
#include "launch.cuh"
#include "pull.cuh"

namespace elbm {

// Nodes are dealt out in a row, 64 to a block: no lane is lost to the ends of rows, small lattices
// reach all SMs, and the node's coordinates (two divisions) are worked out while the launch waits for
// the one before.  Against blocks of 256 that each took pieces of rows (whole passes: steps, start
// and read-outs): 24^3 FP32 plume 171 -> 127 us, 48 x 40 x 32 FP32 at rest 364 -> 352 us (100 steps),
// 121 x 75 x 50 FP32 porous 1043 -> 962 us, 190 x 200 x 180 FP32 porous 3.59 -> 3.16 ms, 200 x 200 x
// 190 FP16 plume 3.04 -> 2.70 ms.  With the divisions after the wait 24^3 137, at rest 422 us; blocks
// of 128 then 141 and 396 us.
constexpr int THREADS = 64;

// Resident warps per SM requested from the register allocator, in units of 8.
#ifndef ELBM_STEP_MINB
#define ELBM_STEP_MINB 3
#endif
// FP64 in fixed point: 34 KB of shared memory per 64 nodes (fixed.cuh) lets 6 blocks stand on an SM
// at 168 registers.  Measured on the 96 x 80 x 72 plume, 20 steps and their read-outs: 4 blocks 4.02,
// 6 blocks 3.54 ms; all loops unrolled, no shared memory, 2 to 4 blocks of 128 3.97 to 4.24 ms
// (waiting for instructions); FP64 arithmetic 10.7 ms.
// FEW: lattices whose blocks stand on the chip 4 to an SM take the registers that 6 would not leave
// them; their time is a node's chain, not throughput.  A step of 32^3 nodes with a plume two nodes
// wide (mostly left to FP64) 77 -> 53 us (FP64 arithmetic alone 54), 5.3 wide 18.5 -> 15 us; 40^3, 6.6
// blocks to an SM, takes 127 us (4 blocks) and 129 us, later 122 and 102 us.
#ifndef ELBM_FIXED_MINB
#define ELBM_FIXED_MINB 6
#endif
constexpr int FEW_PER_SM = 4;
constexpr size_t FEW_NODES = 152ull * FEW_PER_SM * THREADS;
template <typename Elem, int MODE, bool FEW>
__host__ __device__ constexpr int step_blocks() {
  return MODE == FIXED ? (FEW ? FEW_PER_SM : ELBM_FIXED_MINB) : (std::is_same<Elem, double>::value ? 1 : ELBM_STEP_MINB) * (256 / THREADS);
}

template <int MODE>
using Kept = typename std::conditional<MODE == FIXED, InShared<THREADS>, KeepNone>::type;

template <typename Elem, int VEL, int MODE, bool FEW>
__global__ void __launch_bounds__(THREADS, step_blocks<Elem, MODE, FEW>())
k_step(Field<Elem> in, Elem* __restrict__ pout, float* __restrict__ sout, Grid G,
       const typename Storage<Elem>::real* __restrict__ T6,
       const float* __restrict__ src, const float* __restrict__ u3, int fallback,
       unsigned long long* __restrict__ counters, const PopConsts<typename Storage<Elem>::real> k,
       const __grid_constant__ StepConsts<MODE> c) {
  using R = typename Storage<Elem>::real;
  const unsigned m = blockIdx.x * (unsigned)THREADS + threadIdx.x, row = m / (unsigned)G.nx;
  const int x = (int)(m - row * (unsigned)G.nx), y = (int)(row % (unsigned)G.ny), z = (int)(row / (unsigned)G.ny);
  __shared__ int64_t kept[MODE == FIXED ? KEPT * THREADS : 1];
  wait_for_previous();
  bool took = false, proj = false;
  Lanes lanes{};
  if constexpr (MODE == FIXED) lanes = Lanes{__ballot_sync(0xffffffffu, z < G.nz), G.nx};
  if (z < G.nz) {
    const int n = (int)m;
    R g[Q];
    pull_node<Elem, R>(g, in, G, x, y, z, k);
    // merged Strang half-steps of consecutive steps (Section 3.3)
    const R r = src != nullptr ? k.src_step * R(__ldg(src + n)) : R(0);
    const Sym6<R> T = load_T<R>(T6, G.N, n, k.T);
    Kept<MODE> keep{};
    if constexpr (MODE == FIXED) keep = Kept<MODE>{kept + threadIdx.x};
    if constexpr (VEL == 2) {
      const R un[3] = {R(__ldg(u3 + n)), R(__ldg(u3 + G.N + n)), R(__ldg(u3 + 2 * G.N + n))};
      took = collide_and_store<R, VEL, MODE>(g, in, pout, sout, G, n, T, T6 != nullptr, r, src, k, c,
                                             fallback != 0, lanes, keep, proj, un);
    } else {
      took = collide_and_store<R, VEL, MODE>(g, in, pout, sout, G, n, T, T6 != nullptr, r, src, k, c,
                                             fallback != 0, lanes, keep, proj);
    }
  }
  // one counter update per block
  const int cnt = __syncthreads_count(took);
  if (cnt != 0 && threadIdx.x == 0) atomicAdd(counters, (unsigned long long)cnt);
  if constexpr (Storage<Elem>::dev) {
    const int p = __syncthreads_count(proj);
    if (p != 0 && threadIdx.x == 0) atomicAdd(counters + 3, (unsigned long long)p);
  }
}

template <typename Elem, int VEL, int MODE>
static cudaError_t launch_t(const StepLaunch& L, cudaStream_t s) {
  using R = typename Storage<Elem>::real;
  Field<Elem> in{static_cast<const Elem*>(L.pin), L.sin};
  Grid G{L.nx, L.ny, L.nz, L.N, L.dirichlet};
  const PopConsts<R>& k = *reinterpret_cast<const PopConsts<R>*>(std::is_same<R, double>::value ? (const void*)L.kd
                                                                                               : (const void*)L.kf);
  const dim3 blocks((unsigned)((L.N + THREADS - 1) / THREADS));
  auto kernel = k_step<Elem, VEL, MODE, false>;
  if constexpr (MODE == FIXED) {
    if (L.N <= FEW_NODES) kernel = k_step<Elem, VEL, MODE, true>;
  }
  return launch_next(kernel, blocks, dim3(THREADS), 0, s, in, static_cast<Elem*>(L.pout), L.sout, G,
                     static_cast<const R*>(L.T6), L.src, L.u3, L.fallback, L.counters, k, step_consts<MODE>(L));
}

template <typename Elem>
static cudaError_t launch_v(const StepLaunch& L, cudaStream_t s) {
  // the exact root applies only where u != 0 (kappa = 0 at u = 0)
  const bool root = (std::is_same<Elem, double>::value ? L.kd->root : L.kf->root) != 0;
  if (L.vel == 2) return root ? launch_t<Elem, 2, ROOT>(L, s) : launch_t<Elem, 2, CLOSED>(L, s);
  if (L.vel == 1 && root) return launch_t<Elem, 1, ROOT>(L, s);
  if constexpr (std::is_same<Elem, double>::value) {
    if (L.fix->ok) return L.vel == 1 ? launch_t<Elem, 1, FIXED>(L, s) : launch_t<Elem, 0, FIXED>(L, s);
  }
  return L.vel == 1 ? launch_t<Elem, 1, CLOSED>(L, s) : launch_t<Elem, 0, CLOSED>(L, s);
}

int step_variant(int prec, int nx, int vel, bool root, int requested) {
  if (requested != 0) return requested;
  // auto: the staged-row kernel for the FP32-arithmetic storages with rows of 256 nodes or more
  // (uniform velocity, closed-form stabilizer), else the per-node kernel.  Measured, ms/step
  // per-node -> staged: 256^3 plume FP32 0.684 -> 0.588, BF16 deviations 0.782 -> 0.769, FP16
  // deviations 0.777 -> 0.779 (before the deviation kernels' spill fix); 384^3 heterogeneous
  // (tensor field, source, Dirichlet) FP32 2.83 -> 2.48, FP16 2.88 -> 2.35; 320 x 256 x 256 (row
  // length not compiled in) FP32 0.90 -> 0.72, FP16 1.00 -> 0.85.  Kept on the per-node kernel:
  // rows shorter than a block (192^3: FP32 0.256 vs 0.279, FP16 0.279 vs 0.344), per-node
  // velocity fields (256^3: FP32 1.23 vs 1.65, FP16 1.37 vs 1.77; the per-node tables need the
  // registers the staged kernel's persistent loop holds) and FP64 (arithmetic-bound).
  if (prec != 0 && nx >= 256 && vel != 2 && !root && rows_eligible(prec, nx)) return 2;
  return 1;
}

cudaError_t launch_step(const StepLaunch& L, cudaStream_t s) {
  const bool root = (L.prec == 0 ? L.kd->root : L.kf->root) != 0;
  const int v = step_variant(L.prec, L.nx, L.vel, root, L.variant);
  if (v == 3) return launch_step_pipe(L, s);
  if (v == 2)
    return rows_eligible(L.prec, L.nx) ? launch_step_rows(L, s) : cudaErrorNotSupported;
  switch (L.prec) {
    case 0: return launch_v<double>(L, s);
    case 1: return launch_v<float>(L, s);
    case 2: return launch_v<__half>(L, s);
    case 3: return launch_v<__nv_bfloat16>(L, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace elbm
