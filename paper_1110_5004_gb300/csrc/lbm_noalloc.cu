// Allocation-free variant of the FP64 diagnostics reduction.
//
// Who needs it: a caller that cannot call cudaMalloc, because the host application already
// owns the device memory (a server that has reserved the whole budget for its own pools, or a
// solver loop that must not take the implicit device-wide synchronisation of a fresh
// allocation), can still reduce fields it holds.  It passes the four input fields and the
// output record; the partial sums live in a fixed file-scope device array instead of
// memory the library would allocate.
//
// The array is shared by every call in the process on a given device and keeps the last
// call's contents.  Every partial a call reads is written earlier by the same call, and the count of
// finished blocks is cleared by it; two calls whose kernels overlap on the GPU (different streams, no
// ordering between them) race on both and must not be issued: the record of either may be a mixture, or
// an earlier call's.
#include <math.h>
#include <mutex>

#include "lbm_diag.cuh"
#include "lbm_internal.h"

namespace lbm {

constexpr int NOALLOC_MAX_ROWS = 8192;
constexpr int NOALLOC_MAX_DEVICES = 64;

// 8192 rows x 12 partials + the 12-double result record: 768 KB held by every GPU that loads
// the library, until the process exits.
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_MAX_ROWS * DIAG_PARTIALS + 16];

// Device address of the scratch array, looked up once per device with that device current.
static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

static int noalloc_scratch(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_diagnostics_fields_noalloc: cudaGetDevice");
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
    set_error("lbm_diagnostics_fields_noalloc: device %d beyond the %d supported", dev, NOALLOC_MAX_DEVICES);
    return LBM_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    double* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) return cuda_fail(e, "lbm_diagnostics_fields_noalloc: cudaGetSymbolAddress");
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return LBM_OK;
}

// Memory the current device's kernels can address: managed memory, or device memory of this
// device (a field on another GPU would need peer access the library does not set up).
static bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev);
}

}  // namespace lbm

using namespace lbm;

extern "C" int lbm_diagnostics_fields_noalloc(const float* phi, const float* ux, const float* uy, const float* p,
                                              int nx, int ny, double phi_star, long long step, void* cuda_stream,
                                              lbm_diag* out) {
  if (!phi || !ux || !uy || !p || !out) return set_error("fields and out are required"), LBM_ERR_INVALID_ARG;
  if (nx < 1 || ny < 1) return set_error("grid %dx%d is empty", nx, ny), LBM_ERR_INVALID_ARG;
  if (ny > NOALLOC_MAX_ROWS) {
    set_error("lbm_diagnostics_fields_noalloc: ny = %d exceeds the fixed scratch of %d rows", ny, NOALLOC_MAX_ROWS);
    return LBM_ERR_INVALID_ARG;
  }
  if (!(phi_star > 0)) return set_error("phi_star must be positive"), LBM_ERR_INVALID_ARG;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_diagnostics_fields_noalloc: cudaGetDevice");
  if (!on_device(phi, dev) || !on_device(ux, dev) || !on_device(uy, dev) || !on_device(p, dev))
    return set_error("lbm_diagnostics_fields_noalloc: fields must be memory of the current device"),
           LBM_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const bool host_out = !on_device(out, dev);
  if (host_out) {
    // a host record needs a stream synchronisation, which a stream under capture refuses
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(st, &cs)) != cudaSuccess)
      return cuda_fail(e, "lbm_diagnostics_fields_noalloc: cudaStreamIsCapturing");
    if (cs != cudaStreamCaptureStatusNone)
      return set_error("lbm_diagnostics_fields_noalloc: a host out cannot be filled on a capturing stream; "
                       "pass a device out"), LBM_ERR_INVALID_ARG;
  }
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return cuda_fail(e, "lbm_diagnostics_fields_noalloc: device query");
  double* scratch = nullptr;
  int rc = noalloc_scratch(&scratch);
  if (rc) return rc;
  double* record = scratch + (long long)NOALLOC_MAX_ROWS * DIAG_PARTIALS;
  // the count of finished blocks is cleared by each call: an earlier one may have been cut short
  unsigned int* done = reinterpret_cast<unsigned int*>(record + 15);
  if ((e = cudaMemsetAsync(done, 0, sizeof(unsigned int), st)) != cudaSuccess)
    return cuda_fail(e, "lbm_diagnostics_fields_noalloc: block count");
  e = launch_diag_rows(diag_in(phi, ux, uy, p, nx, ny, nx, phi_star, scratch, record, done, step), sms, st);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_diagnostics_fields_noalloc: kernel");
  e = cudaMemcpyAsync(out, record, sizeof(lbm_diag), host_out ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && host_out) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_diagnostics_fields_noalloc: result copy");
  if (host_out && !out->finite) {
    set_error("fields are not finite (step %lld)", step);
    return LBM_ERR_DIVERGED;
  }
  return LBM_OK;
}
