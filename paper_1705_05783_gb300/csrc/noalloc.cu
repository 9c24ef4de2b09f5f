// Residual and 2-norm of a 7-point system with no device allocation.
//
// Some callers cannot call cudaMalloc: frameworks that hand all device memory
// to their own pool or arena (a cudaMalloc behind the pool's back can fail or
// fragment it), and time-critical loops that must not pay the device-wide
// synchronisation that cudaMalloc/cudaFree imply.  This entry point serves
// them: the caller passes the system and the output buffers, and the
// reduction's scratch (one partial sum per CTA plus the total)
// lives in a file-scope static device array instead of a handle allocation.
//
// The array exists once per device that loads the library and stays there
// until the process exits.  In host code its name is only a host-side stand-in,
// so its device address is looked up with cudaGetSymbolAddress, with the
// device current: on the first call on a device, and again whenever the
// device's current context differs from the one the address was taken in (the
// module is loaded anew after cudaDeviceReset, and the array may move).
// Every call shares the array: calls that overlap on the GPU (different
// streams, or several host threads) race on it and must be serialised by the
// caller.  Each call overwrites every slot it reads, so nothing left by an
// earlier call leaks into a result.
#include <atomic>
#include <cmath>
#include <mutex>
#include <string>
#include <utility>

#include <cooperative_groups.h>

#include "cams_internal.h"
#include "launch.h"
#include "stencil.h"

namespace {

// the entry point's limit, part of its contract (no buffer here depends on it)
constexpr long long kMaxCells = 1LL << 28;   // 268,435,456

// A grid of at most kSmallPieces pieces of kSmallThreads columns goes to one
// cluster, whose CTAs sum up through distributed shared memory: the second
// launch that adds the partial sums would cost as much as the residual.  (A
// call on 40 x 40 cells: 23 us, of which 6 are the caller's Python; 36 with two
// launches and a copy of the total.  On 32 x 32 x 32 cells, the largest of the
// rule, 26 against 29.)
constexpr int kSmallThreads = 1024, kSmallCtas = 8, kSmallPieces = 4 * kSmallCtas;
constexpr int kMaxDevices = 64;

// one partial sum per CTA, then the total
static __device__ __align__(256) double g_noalloc_scratch[cams::kColBlocks + 1];

std::mutex g_mutex;
double* g_scratch_addr[kMaxDevices] = {};
unsigned long long g_scratch_ctx[kMaxDevices] = {};   // context the address was taken in

__global__ void __launch_bounds__(cams::kColThreads) k_residual_noalloc(
    cams::Geo g, cams::ColWork w, const double* __restrict__ Ad, const double* __restrict__ Ax,
    const double* __restrict__ Ay, const double* __restrict__ Az, const double* __restrict__ f,
    const double* __restrict__ p, double* r, double* scratch) {
  const double s2 = cams::block_sum(
      cams::residual_columns(g, w, Ad, Ax, Ay, Az, Ax, Ay, Az, f, p, r, nullptr));
  if (threadIdx.x == 0) scratch[blockIdx.x] = s2;
}

// The whole residual and its total by one cluster of CTAs.
__global__ void __launch_bounds__(kSmallThreads) k_residual_small(
    cams::Geo g, cams::ColWork w, const double* __restrict__ Ad, const double* __restrict__ Ax,
    const double* __restrict__ Ay, const double* __restrict__ Az, const double* __restrict__ f,
    const double* __restrict__ p, double* r, double* total) {
  __shared__ double part[kSmallCtas];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  // (CTA 0's shared memory is written once it is known to have started)
  auto started = cl.barrier_arrive();
  const double s2 = cams::block_sum(
      cams::residual_columns(g, w, Ad, Ax, Ay, Az, Ax, Ay, Az, f, p, r, nullptr));
  cl.barrier_wait(std::move(started));
  if (threadIdx.x == 0) cl.map_shared_rank(part, 0)[blockIdx.x] = s2;
  cl.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double s = 0.0;
    for (int b = 0; b < (int)gridDim.x; ++b) s += part[b];
    *total = s;
  }
}

// total of the partial sums, in block order (deterministic)
__global__ void k_finish_noalloc(int nblocks, const double* scratch, double* total) {
  double s = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) s += scratch[b];
  s = cams::block_sum(s);
  if (threadIdx.x == 0) *total = s;
}

// Whether the device can hold k_residual_small's clusters (asked once).
bool small_fits(int dev) {
  static std::atomic<int> known[kMaxDevices];   // 0 not asked, 1 no, 2 yes
  int k = known[dev].load(std::memory_order_relaxed);
  if (k == 0) {
    k = cams::cluster_fits(k_residual_small, kSmallCtas, kSmallThreads, 0) ? 2 : 1;
    known[dev].store(k, std::memory_order_relaxed);
  }
  return k == 2;
}

int fail_na(int code, const std::string& msg) {
  cams::set_global_error(msg);
  return code;
}

}  // namespace

namespace cams {

// The driver's number of the calling thread's current context, unique in the
// process (a device's context keeps its handle over cudaDeviceReset, but not its
// number); 0 when there is none or it cannot be told.  cuCtxGetCurrent and
// cuCtxGetId are reached through the runtime (no link against libcuda); a
// CUcontext is held as an opaque pointer.
unsigned long long context_id() {
  using GetCurrent = int (*)(void**);
  using GetId = int (*)(void*, unsigned long long*);
  static const auto entry = [](const char* name) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion(name, &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      fn = nullptr;
    }
    return fn;
  };
  static const auto get = reinterpret_cast<GetCurrent>(entry("cuCtxGetCurrent"));
  static const auto id_of = reinterpret_cast<GetId>(entry("cuCtxGetId"));
  void* ctx = nullptr;
  unsigned long long id = 0;
  if (!get || !id_of || get(&ctx) != 0 || !ctx || id_of(ctx, &id) != 0) return 0;
  return id;
}

// Whether kernels on the device can write ordinary host memory.
bool host_writable(int dev) {
  static std::atomic<int> known[kMaxDevices];   // 0 not asked, 1 no, 2 yes
  if (dev < 0 || dev >= kMaxDevices) return false;
  int k = known[dev].load(std::memory_order_relaxed);
  if (k == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev) != cudaSuccess) v = 0;
    k = v ? 2 : 1;
    known[dev].store(k, std::memory_order_relaxed);
  }
  return k == 2;
}

}  // namespace cams

extern "C" int cams_residual_norm_noalloc(int nx, int ny, int nz, const double* diag,
                                          const double* ax, const double* ay, const double* az,
                                          const double* f, const double* p, double* r,
                                          double* norm_out, void* stream) {
  if (nx < 1 || ny < 1 || nz < 1) return fail_na(CAMS_EINVAL, "grid sizes must be >= 1");
  const long long N = (long long)nx * ny * nz;
  if (N > kMaxCells)
    return fail_na(CAMS_EINVAL, "cams_residual_norm_noalloc: the grid has " + std::to_string(N) +
                                    " cells; at most " + std::to_string(kMaxCells) +
                                    " are supported");
  if (!diag || !ax || !ay || !az || !f || !p) return fail_na(CAMS_EINVAL, "null input pointer");
  if (!r && !norm_out) return fail_na(CAMS_EINVAL, "no output requested");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_na(CAMS_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail_na(CAMS_EINVAL, "device ordinal out of range");
  double* scratch = nullptr;
  {
    // set-up, once per device and context, with that device current
    std::lock_guard<std::mutex> lock(g_mutex);
    const unsigned long long ctx = cams::context_id();
    if (!g_scratch_addr[dev] || !ctx || ctx != g_scratch_ctx[dev]) {
      e = cudaGetSymbolAddress(reinterpret_cast<void**>(&scratch), g_noalloc_scratch);
      if (e != cudaSuccess)
        return fail_na(CAMS_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      g_scratch_addr[dev] = scratch;
      g_scratch_ctx[dev] = cams::context_id();   // the lookup made the primary context current
    }
    scratch = g_scratch_addr[dev];
  }
  cams::Geo g{};
  g.nx = nx; g.ny = ny; g.nz = nz;
  g.N = N;
  g.sy = nx; g.sz = (long long)nx * ny;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // Where the GPU can write this thread's stack (it shares the host's page
  // tables), the total goes straight to it and the stream's end makes it
  // visible; a copy of the eight bytes takes 5 to 10 us more.  So nothing below
  // returns before the stream is done, and a launch is judged by its own code: an
  // earlier call's error, still pending in the runtime, is not this one's.
  double s2 = 0.0;
  const bool direct = norm_out && cams::host_writable(dev);
  double* total = direct ? &s2 : scratch + cams::kColBlocks;
  const char* what = "launch: ";
  cams::ColWork w = cams::col_work(g, kSmallThreads);
  if (w.pieces <= (unsigned)kSmallPieces && small_fits(dev)) {
    int ctas = 1;
    while (ctas < kSmallCtas && ctas < (int)w.pieces) ctas *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctas > 1 ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, k_residual_small, g, w, diag, ax, ay, az, f, p, r, total);
    cams::count_launches(1);
  } else {
    w = cams::col_work(g);
    const int nblocks = cams::col_grid(w);
    e = cams::launch_after(false, k_residual_noalloc, dim3(nblocks), cams::kColThreads, 0, s, g, w, diag,
                           ax, ay, az, f, p, r, scratch);
    if (e == cudaSuccess)
      e = cams::launch_after(false, k_finish_noalloc, dim3(1), 1024, 0, s, nblocks, scratch, total);
    cams::count_launches(2);
  }
  if (e == cudaSuccess && norm_out && !direct) {
    what = "read-back: ";
    e = cudaMemcpyAsync(&s2, total, sizeof(double), cudaMemcpyDeviceToHost, s);
  }
  const cudaError_t done = cudaStreamSynchronize(s);
  if (e == cudaSuccess) {
    what = "synchronize: ";
    e = done;
  }
  if (e != cudaSuccess) return fail_na(CAMS_ECUDA, std::string(what) + cudaGetErrorString(e));
  if (norm_out) *norm_out = std::sqrt(*static_cast<volatile double*>(&s2));
  return CAMS_OK;
}
