// Conservation diagnostics of a caller-held population state without any device
// allocation: the reduction of reduce.cuh with its partial sums in a file-scope device
// array instead of a buffer from cudaMalloc.
//
// Who needs it: code that must not allocate device memory at the moment it wants
// the diagnostics -- a process whose device memory is already fully reserved by
// another allocator (a framework's caching allocator or a memory pool that owns the
// GPU), or a monitoring hook inside a time-stepping loop where an allocation that
// blocks or fails is not acceptable (e.g. reporting after an out-of-memory error).
#include <cmath>
#include <mutex>

#include "../../include/elbm.h"
#include "internal.h"
#include "reduce.cuh"

using namespace elbm;

namespace {

constexpr int kMaxPartials = 4096;  // blocks of the partial-sum kernel that the array has room for
static_assert(REDUCE_BLOCKS <= kMaxPartials, "partial sums fit the fixed array");
constexpr int kMaxDevices = 64;

// 4 doubles per block (mass, entropy, min g, non-finite count) + 4 for the final result:
// 131 104 bytes on every GPU that loads the library, held until the process exits.
__device__ __align__(256) double g_scratch[4 * kMaxPartials + 4];

std::mutex g_mu;
// Device address of g_scratch per device, and the id of the context it was looked up in: a
// module's __device__ arrays are placed anew when a device's context is destroyed and
// re-created (cudaDeviceReset), so the address is looked up again when the id changes.
double* g_scratch_dev[kMaxDevices] = {};
unsigned long long g_scratch_ctx[kMaxDevices] = {};

// Unique id of the current context (driver entry points fetched through the runtime, so the
// library needs no link against the driver library); 0 if it cannot be had.
unsigned long long current_context_id() {
  typedef int (*get_current_t)(void**);
  typedef int (*get_id_t)(void*, unsigned long long*);
  static get_current_t get_current = nullptr;
  static get_id_t get_id = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    cudaDriverEntryPointQueryResult q1, q2;
    void* f1 = nullptr;
    void* f2 = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
        q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
      get_current = reinterpret_cast<get_current_t>(f1);
      get_id = reinterpret_cast<get_id_t>(f2);
    }
    cudaGetLastError();
    looked_up = true;
  }
  void* ctx = nullptr;
  unsigned long long id = 0;
  if (get_current && get_id && get_current(&ctx) == 0 && ctx != nullptr && get_id(ctx, &id) == 0) return id;
  return 0;
}

// Device address of g_scratch on the current device: looked up (cudaGetSymbolAddress, with
// the device current) on the first call in each context of that device, then cached.
cudaError_t scratch_address(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mu);
  const unsigned long long ctx = current_context_id();
  if (g_scratch_dev[dev] == nullptr || ctx == 0 || ctx != g_scratch_ctx[dev]) {
    double* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_dev[dev] = p;
    // the symbol lookup made the runtime create the context if there was none yet
    g_scratch_ctx[dev] = ctx != 0 ? ctx : current_context_id();
  }
  *out = g_scratch_dev[dev];
  return cudaSuccess;
}

template <typename R>
PopConsts<R> pull_consts(const double u[3], const elbm_bc* bc) {
  PopConsts<R> k{};
  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  for (int i = 0; i < Q; ++i) {
    const double cu = cx_of(i) * u[0] + cy_of(i) * u[1] + cz_of(i) * u[2];
    k.E[i] = (R)(w_of(i) * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu));
  }
  k.phi_lo = (R)(bc ? bc->phi_lo : 0.0);
  k.phi_hi = (R)(bc ? bc->phi_hi : 0.0);
  return k;
}

template <typename Elem>
cudaError_t launch(const void* pops, const float* scale, const Grid& G, const float* src, const double u[3],
                   const elbm_bc* bc, double* scratch, double* out4, cudaStream_t s) {
  using R = typename Storage<Elem>::real;
  Field<Elem> f{static_cast<const Elem*>(pops), scale};
  return launch_reduce_t<Elem>(f, G, src, 0.5, scratch, out4, pull_consts<R>(u, bc), s);
}

bool device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" elbm_status elbm_reduce_noalloc(const void* pops, const float* scale, const int64_t dims[3],
                                           elbm_precision prec, const double u[3], const elbm_bc* bc,
                                           const float* source, void* cuda_stream, double out4[4]) {
  if (!pops || !dims || !u || !out4) return ELBM_ERR_ARG;
  if ((int)prec < 0 || (int)prec > 3) return ELBM_ERR_ARG;
  if (prec >= ELBM_F32_F16DEV && !scale) return ELBM_ERR_ARG;
  // the kernels read these directly: a host pointer here would make them fault
  if (!device_ptr(pops) || (prec >= ELBM_F32_F16DEV && !device_ptr(scale)) || (source && !device_ptr(source)))
    return ELBM_ERR_ARG;
  for (int a = 0; a < 3; ++a)
    if (dims[a] < 1 || dims[a] > 65535) return ELBM_ERR_ARG;
  const double N = (double)dims[0] * (double)dims[1] * (double)dims[2];
  if (27.0 * N >= 2147483647.0) return ELBM_ERR_ARG;  // same lattice limit as elbm_create
  if (bc && bc->dirichlet_x != 0 && bc->dirichlet_x != 1) return ELBM_ERR_ARG;
  double* scratch = nullptr;
  if (scratch_address(&scratch) != cudaSuccess) return ELBM_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  Grid G{(int)dims[0], (int)dims[1], (int)dims[2], (size_t)N, bc ? bc->dirichlet_x : 0};
  const bool host_out = !device_ptr(out4);
  double* dst = host_out ? scratch + 4 * kMaxPartials : out4;
  cudaError_t e = cudaErrorInvalidValue;
  switch ((int)prec) {
    case 0: e = launch<double>(pops, scale, G, source, u, bc, scratch, dst, s); break;
    case 1: e = launch<float>(pops, scale, G, source, u, bc, scratch, dst, s); break;
    case 2: e = launch<__half>(pops, scale, G, source, u, bc, scratch, dst, s); break;
    case 3: e = launch<__nv_bfloat16>(pops, scale, G, source, u, bc, scratch, dst, s); break;
  }
  if (e != cudaSuccess) return ELBM_ERR_CUDA;
  if (host_out) {
    if (cudaMemcpyAsync(out4, dst, 4 * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess) return ELBM_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return ELBM_ERR_CUDA;
  }
  return ELBM_OK;
}
