// re_noalloc.cu -- LJ forces of caller-given positions without any device or
// host allocation, for callers that cannot call cudaMalloc.
//
// Some callers cannot allocate device memory: code that runs inside another
// framework's memory pool or under a fixed memory budget, a plug-in that may
// not touch the allocator, or a path that must not add allocation latency.
// re_lj_forces_device_noalloc serves them: it computes what
// re_lj_forces_device computes (FP64 pair forces, the same kernels) but keeps
// the intermediate arrays (fixed-point positions, partial energies, status) in
// one file-scope device array, g_scratch, of fixed size.
//
// Limits: N <= kMaxAtoms atoms and at most kMaxNeighbours atoms within the list
// radius rc + 0.5 of one (density times that sphere's volume, with margin).  The
// array lives on every device that loads this library until the process exits.
// The first call on a device looks up the array's device address
// (cudaGetSymbolAddress) and caches it; make that first call before any
// stream capture.  All calls share the array: it keeps the previous call's
// contents, the call clears what must start at zero, and calls that overlap
// on the GPU (different streams, or threads without ordering) race.
#include <cuda_runtime.h>

#include <atomic>

#include "re.h"
#include "re_internal.h"

namespace {

constexpr int kMaxAtoms = 4096;
constexpr int kMaxNeighbours = 256;
constexpr int kMaxDevices = 64;
constexpr size_t kScratch = (size_t)kMaxAtoms * 56 + ((size_t)kMaxAtoms / 4 + 2) * 8;

// device address of g_scratch, per device; every thread that fills an entry
// stores the same value, so relaxed atomic accesses suffice
std::atomic<void*> g_scratch_dev[kMaxDevices];

// errors are reported by return code only (a message would need allocation)
int fail(int code, const char*) { return code; }

}  // namespace

// The scratch array: one per device that loads the library, for its lifetime.
static __device__ __align__(256) unsigned char g_scratch[kScratch];

extern "C" int re_lj_forces_device_noalloc(int N, double L, double rc, int shift, const double* x,
                                           double* f, double* U, void* stream) {
  if (N < 2 || N > kMaxAtoms) return fail(RE_EINVAL, "N must be in [2, 4096]");
  if (!x || !f || !U) return fail(RE_EINVAL, "NULL device pointer");
  if (!(L > 0) || !(rc > 0) || rc + 0.5 >= 0.5 * L) return fail(RE_EINVAL, "need rc + 0.5 < L/2");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(RE_ECUDA, "no usable current device");
  // once per device, with that device current: the array's device address
  void* sp = g_scratch_dev[dev].load(std::memory_order_relaxed);
  if (!sp) {
    const cudaError_t e = cudaGetSymbolAddress(&sp, g_scratch);
    if (e != cudaSuccess || !sp) return fail(RE_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
    g_scratch_dev[dev].store(sp, std::memory_order_relaxed);
  }
  if (re::direct_scratch_bytes(N) > kScratch) return fail(RE_EINVAL, "scratch array too small");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int sms = 0;
  cudaError_t ce = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (ce != cudaSuccess) return fail(RE_ECUDA, cudaGetErrorString(ce));

  // the ensemble's constants (list radius rc + 0.5)
  re::EnsDev e{};
  e.N = N;
  e.R = 1;
  e.L = L;
  e.rc = rc;
  e.skin = 0.5;
  e.rlist = rc + 0.5;
  e.dt = 0.005;
  e.tau = 0.0;
  e.shift = shift ? 1 : 0;
  re::set_capacity(e, 0);
  re::finish_ens(e);
  if (e.capsub[0] > kMaxNeighbours)
    return fail(RE_EOVERFLOW, "density too high for the fixed neighbour capacity (256 per atom)");
  int32_t* d_status = nullptr;
  int32_t status = 0;
  if ((ce = re::launch_lj_direct(sp, N, e.kc, false, e.capsub[0], sms, x, f, U, &d_status, st)) ||
      (ce = cudaMemcpyAsync(&status, d_status, sizeof status, cudaMemcpyDeviceToHost, st)) ||
      (ce = cudaStreamSynchronize(st)))
    return fail(RE_ECUDA, cudaGetErrorString(ce));
  if (status & re::kStOverflow) return fail(RE_EOVERFLOW, "neighbour list capacity exceeded");
  if (status) return fail(RE_ENUMERIC, "non-finite energy (overlapping atoms?)");
  return RE_OK;
}
