// Allocation-free misfit reduction: ddfd_misfit_noalloc.
//
// Who needs it: callers that must not allocate device memory -- for example
// code running under a strict memory budget or inside a host framework that
// owns every device allocation (a custom allocator, a pre-planned arena, a
// real-time loop where cudaMalloc's implicit synchronisation and latency are
// not acceptable).  Such a caller cannot create a ddfd handle, because
// ddfd_create allocates the field buffers; this entry point needs no handle.
//
// Its only scratch is the file-scope array below: one FP64 partial sum per
// (source, time step) row of the trace.  It is part of the library image,
// so every GPU that loads the library holds it (512 KB) until the process
// exits; no call allocates or frees anything.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>
#include <string>

#include "ddfd_internal.h"
#include "ddfd_tma.h"

namespace ddfd {
void set_thread_error(const std::string &msg);
}

namespace {

constexpr int kNoallocMaxRows = 65536;  // n_src * (n_steps + 1) at most
constexpr int kRB = 256;

static __device__ __align__(256) double g_misfit_rows[kNoallocMaxRows];

// Sum over the block's NT threads, valid in thread 0.
template <int NT>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[NT / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (l < NT / 32) ? sh[l] : 0.0;
    for (int o = NT / 64; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  __syncthreads();
  return v;
}

// Pass 1: rows[s (n_steps+1) + n] = z(t_n) sum_d |trace - eobs|^2 (0 for n = 0).
// Every row in [0, n_rows) is written, so the scratch needs no clearing.  GROUP
// threads sum a row: a warp for short rows (eight rows a thread block), else
// the block.  What bounds the small sizes is the FP64 unit's latency (64 cycles
// an instruction and warp, whatever its lanes): the taper's cosine is evaluated
// only in the rows that it touches, t > ramp = T - dl (inv_dl = 1 / dl; ramp is
// infinite without a taper), by one warp.  Its phase is formed as (t - T) + dl, whose
// first difference is exact: t - ramp would carry the rounding of T - dl, an error of
// 1e-16 T / dl in the phase of a short taper.  Large sizes are bound by the FP64
// unit's rate (two instructions a value).  us a call, before (a thread block per
// row, two plain launches) and now: 300 steps x 64 detectors 12.3 -> 8.2 (6.8 of
// it on the host), 2000 x 1024 57 -> 38, 8 sources of it 337 -> 245.
template <int GROUP>
__global__ void __launch_bounds__(kRB) k_misfit_rows(const double *__restrict__ trace, const double *__restrict__ eobs,
                                                     int n_steps, int n_det, int n_rows, double tau, double T,
                                                     double dl, double ramp, double inv_dl, double *rows) {
  ddfd::pdl_launch_dependents();
  constexpr int PER = kRB / GROUP;
  const int g = threadIdx.x / GROUP, l = threadIdx.x % GROUP;
  for (int row = blockIdx.x * PER + g; row < n_rows; row += gridDim.x * PER) {
    const int step = row % (n_steps + 1);
    const double *tr = trace + (long long)row * n_det * 3, *eo = eobs + (long long)row * n_det * 3;
    const int nv = step >= 1 ? 3 * n_det : 0;
    double acc = 0.0;
    int q = l;
    for (; q + 3 * GROUP < nv; q += 4 * GROUP) {  // four values a thread in flight
      double d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = tr[q + i * GROUP] - eo[q + i * GROUP];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc += d[i] * d[i];
    }
    for (; q < nv; q += GROUP) {
      const double d = tr[q] - eo[q];
      acc += d * d;
    }
    double z = 1.0;
    if (l < 32) {
      const double t = __dmul_rn((double)step, tau);  // (rounded, as T is: T - T has to be zero)
      if (t > ramp) z = 0.5 * (1.0 + cospi(((t - T) + dl) * inv_dl));
    }
    double b;
    if (GROUP == 32) {
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
      b = acc;
    } else {
      b = block_sum<kRB>(acc);
    }
    if (l == 0) rows[row] = z * b;
  }
}

// Pass 2: J = tau/2 sum of the rows, fixed-order tree (bitwise reproducible).
// A programmatic dependent of pass 1 (its launch overlaps that one's work).
template <int NT>
__global__ void __launch_bounds__(NT) k_misfit_total(const double *rows, int n_rows, double tau, double *J) {
  ddfd::pdl_wait();
  double a = 0.0;
  for (int q = threadIdx.x; q < n_rows; q += NT) a += rows[q];
  const double b = block_sum<NT>(a);
  if (threadIdx.x == 0) *J = 0.5 * tau * b;
}

// Device address of the scratch array.  The array's host-side name is not a
// device address, so it is resolved with cudaGetSymbolAddress, with the
// device current, once per device context: the cache entry of a device is
// keyed on the context's process-unique id (cuCtxGetId), so a context that
// was reset and re-created (cudaDeviceReset) resolves the address again
// instead of reusing a stale one.
typedef CUresult (*PfnCtxGetCurrent)(CUcontext *);
typedef CUresult (*PfnCtxGetId)(CUcontext, unsigned long long *);

std::mutex g_mu;
struct RowsAddr {
  unsigned long long ctx_id = 0;  // 0: not resolved
  double *addr = nullptr;
};
RowsAddr g_rows_addr[64];
PfnCtxGetCurrent g_ctx_current = nullptr;
PfnCtxGetId g_ctx_id = nullptr;

int driver_fn(const char *name, void **fn) {
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !*fn) {
    ddfd::set_thread_error(std::string(name) + " is not available from the driver");
    return DDFD_E_CUDA;
  }
  return DDFD_OK;
}

// Id of the current context (0 if none is current yet).
int current_ctx_id(unsigned long long *id) {
  *id = 0;
  CUcontext ctx = nullptr;
  if (g_ctx_current(&ctx) != CUDA_SUCCESS) {
    ddfd::set_thread_error("cuCtxGetCurrent failed");
    return DDFD_E_CUDA;
  }
  if (ctx && g_ctx_id(ctx, id) != CUDA_SUCCESS) {
    ddfd::set_thread_error("cuCtxGetId failed");
    return DDFD_E_CUDA;
  }
  return DDFD_OK;
}

int rows_address(double **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    ddfd::set_thread_error(std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    return DDFD_E_CUDA;
  }
  if (dev < 0 || dev >= 64) {
    ddfd::set_thread_error("device ordinal out of range");
    return DDFD_E_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_mu);
  int st;
  if (!g_ctx_current && ((st = driver_fn("cuCtxGetCurrent", (void **)&g_ctx_current)) != DDFD_OK ||
                         (st = driver_fn("cuCtxGetId", (void **)&g_ctx_id)) != DDFD_OK)) {
    g_ctx_current = nullptr;
    return st;
  }
  unsigned long long id = 0;
  if ((st = current_ctx_id(&id)) != DDFD_OK) return st;
  RowsAddr &c = g_rows_addr[dev];
  if (id == 0 || c.ctx_id != id) {
    // first use on this device or context: resolving the symbol also makes
    // the device's primary context current if nothing was current yet
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_misfit_rows);
    if (e != cudaSuccess || !p) {
      ddfd::set_thread_error(std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      return DDFD_E_CUDA;
    }
    if (id == 0 && (st = current_ctx_id(&id)) != DDFD_OK) return st;
    c.ctx_id = id;
    c.addr = (double *)p;
  }
  *out = c.addr;
  return DDFD_OK;
}

}  // namespace

extern "C" int ddfd_misfit_noalloc(const double *trace, const double *eobs, int32_t n_src, int32_t n_steps,
                                   int32_t n_det, double tau, double z_delta_frac, double *J, void *stream) {
  if (!J || n_src < 1 || n_steps < 1 || n_det < 0 || !(tau > 0.0) || !(z_delta_frac >= 0.0 && z_delta_frac < 1.0) ||
      (n_det > 0 && (!trace || !eobs))) {
    ddfd::set_thread_error("ddfd_misfit_noalloc: bad argument");
    return DDFD_E_ARG;
  }
  const long long n_rows = (long long)n_src * ((long long)n_steps + 1);
  if (n_rows < 1 || n_rows > kNoallocMaxRows) {
    ddfd::set_thread_error("ddfd_misfit_noalloc: n_src * (n_steps + 1) = " + std::to_string(n_rows) +
                           " exceeds the fixed scratch of " + std::to_string(kNoallocMaxRows) + " rows");
    return DDFD_E_ARG;
  }
  double *rows = nullptr;
  const int st = rows_address(&rows);
  if (st != DDFD_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  const double T = n_steps * tau, dl = z_delta_frac * T;
  const double ramp = dl > 0.0 ? T - dl : HUGE_VAL, inv_dl = dl > 0.0 ? 1.0 / dl : 0.0;
  if (n_det <= 341) {  // up to 32 values a lane: a warp per row
    const long long nb = (n_rows + kRB / 32 - 1) / (kRB / 32);
    k_misfit_rows<32><<<(int)(nb < 4096 ? nb : 4096), kRB, 0, s>>>(trace, eobs, n_steps, n_det, (int)n_rows, tau,
                                                                    T, dl, ramp, inv_dl, rows);
  } else {
    k_misfit_rows<kRB><<<(int)(n_rows < 4096 ? n_rows : 4096), kRB, 0, s>>>(trace, eobs, n_steps, n_det, (int)n_rows,
                                                                            tau, T, dl, ramp, inv_dl, rows);
  }
  if (n_rows <= 2048)
    ddfd::launch_chained(k_misfit_total<kRB>, dim3(1), kRB, 0, s, true, (const double *)rows, (int)n_rows, tau, J);
  else
    ddfd::launch_chained(k_misfit_total<1024>, dim3(1), 1024, 0, s, true, (const double *)rows, (int)n_rows, tau, J);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    ddfd::set_thread_error(std::string("ddfd_misfit_noalloc launch: ") + cudaGetErrorString(e));
    return DDFD_E_CUDA;
  }
  return DDFD_OK;
}
