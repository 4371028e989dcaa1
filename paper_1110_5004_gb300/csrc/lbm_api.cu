// Host runtime and C ABI of liblbm: simulation objects, parameter checks, field transfer,
// step launches and diagnostics.  See include/lbm.h for the contract of every entry point.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <initializer_list>
#include <mutex>
#include <new>
#include <string>

#include "lbm_internal.h"
#include "lbm_march.cuh"

namespace lbm {

static thread_local std::string g_last_error;

void set_error(const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
}

int cuda_fail(cudaError_t e, const char* what) {
  set_error("%s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

Phys make_phys(const lbm_params& p) {
  Phys P{};
  const double cs2 = 1.0 / 3.0;
  const double rho_prime = (p.rho_A - p.rho_B) / (2.0 * p.phi_star);
  P.four_beta = (float)(4.0 * p.beta);
  P.kappa = (float)p.kappa;
  P.phi_star = (float)p.phi_star;
  P.phi_star2 = (float)(p.phi_star * p.phi_star);
  P.inv_2phistar = (float)(1.0 / (2.0 * p.phi_star));
  P.rho_B = (float)p.rho_B;
  P.drho = (float)(p.rho_A - p.rho_B);
  P.ngravity = -(float)p.gravity;
  P.omega_f = (float)(1.0 / p.tau_f);
  P.three_gamma_f = (float)(3.0 * p.theta_M / (p.tau_f - 0.5));
  P.remove_Fa = p.remove_Fa ? 1 : 0;
  P.ch_conv = p.ch_conservative ? 0 : 1;
  P.fs_mu = p.fs_form ? 1 : 0;
  P.s_direct = p.s_form ? 1 : 0;
  P.nkappa6 = -(float)(p.kappa / 6.0);
  P.rho_prime12 = (float)(rho_prime / 12.0);
  P.s_coef6 = (float)(rho_prime * p.theta_M / 6.0);
  P.mu3_B = (float)(3.0 * p.rho_B * cs2 * (p.tau_g_B - 0.5));
  P.mu3_d = (float)(3.0 * (p.rho_A * cs2 * (p.tau_g_A - 0.5) - p.rho_B * cs2 * (p.tau_g_B - 0.5)));
  P.keep_f = (float)(1.0 - 1.0 / p.tau_f);
  P.of3gf = (float)(3.0 * p.theta_M / (p.tau_f - 0.5) / p.tau_f);
  P.f_forced = p.f_form ? 1 : 0;
  P.hf12 = (float)((1.0 - 0.5 / p.tau_f) / 12.0);
  P.thM6 = (float)(p.theta_M / 6.0);
  return P;
}

MarchShape march_shape_of(int nx, int storage, bool sd, int nt) {
  const int slots = march_slots(nt, storage, sd);
  for (int most = nt - 6;;) {
    const int strips = (nx + 2 * most - 1) / (2 * most), width = (nx + 2 * strips - 1) / (2 * strips);
    if (nt < MARCH_NT && width < 16 && strips > 1) return MarchShape{nt, 0, 0};   // more halo than strip
    bool fits = true;
    for (int k = 0; k < strips && fits; ++k) {
      const StagedRun r = staged_run(nx, k * 2 * width, width);
      fits = r.run1 + r.run2 <= slots;
    }
    if (fits) return MarchShape{nt, strips, width};
    most = width - 1;                              // (more strips of the same width stage the same columns)
  }
}

// Rows of a segment: as many segments as fit in one wave of resident CTAs.  The step lasts as long as the
// busiest SM, so a count just above the slots adds a nearly empty wave.  Segments of a few rows spend
// most of their h + 7 iterations on the rows around them, and are still the fastest where the grid has
// no more rows to give (601 x 437 with side walls: 18.1 us at 5 rows, 22.4 at 8)
static int wave_rows(const MarchShape& m, int ny, int sms) {
  const int slots = sms * march_ctas(m.nt), segs = slots >= m.strips ? slots / m.strips : 1;
  return (ny + segs - 1) / segs;
}

// An SM works on the columns of 2 strips of 128-thread CTAs at a time, or of 4 of 64-thread ones, or of 8; a row
// iteration takes as long.  So fewer threads where they shorten a segment's h + 7 iterations by a seventh, else the wider
// strip with its smaller share of halo.  On long grids that is up to 116 columns (whole rows) and 245 to 270 (three
// strips of 90 instead of two) for 64, up to 52 for 32.  us a step, 128 threads -> fewer, FP32 and FP16: 32 x 65536
// 279 -> 82 and 294 -> 80, 64 x 32768 145 -> 79 and 155 -> 76, 100 x 20000 93 -> 69 and 99 -> 51, 250 x 8000 79 -> 65 and
// 82 -> 60; 16 x 16, one row a segment either way, 6.6 -> 7.2.
MarchShape march_shape(int nx, int ny, int storage, bool sd, int sms) {
  MarchShape best = march_shape_of(nx, storage, sd, MARCH_NT);
  for (int nt = MARCH_NT / 2; nt >= 32; nt /= 2) {
    if (nx > 4 * MARCH_NT) break;                  // three strips of 128 threads and more leave nothing to gain
    const MarchShape m = march_shape_of(nx, storage, sd, nt);
    if (m.strips > 0 && 7LL * (wave_rows(m, ny, sms) + 7) < 6LL * (wave_rows(best, ny, sms) + 7)) best = m;
  }
  return best;
}

void tile_geometry(const MarchShape& m, int seg_h, int sms, Grid* g) {
  g->march_nt = m.nt;
  g->n_strips = m.strips;
  g->tile_w = m.width;
  g->seg_h = seg_h <= 0 ? wave_rows(m, g->ny, sms) : std::min(seg_h, g->ny);
}

Grid make_grid(const lbm_sim* s, const void* src, void* dst) {
  Grid g{};
  g.src = src;
  g.dst = dst;
  g.plane = (int)s->plane;
  g.row_bytes = (int)(s->pitch * state_bytes_per_cell(s->params.storage));
  g.nblk = s->pitch / BLK;
  g.storage = s->params.storage;
  g.nx = s->nx;
  g.ny = s->ny;
  g.pitch = s->pitch;
  g.bc_x = s->params.bc_x;
  g.bc_y = s->params.bc_y;
  tile_geometry(s->shape, s->seg_h, s->sms, &g);
  g.wait_tries = (int)std::min(std::max(s->wait_ns, WAIT_LEAST_NS) / WAIT_TRY_NS + 1, 1LL << 30);
  g.wait_hold = -1;
  g.give_up = GiveUp{gave_up(s), s->slot ? &s->slot->gave_up : nullptr};
  g.spoff = s->params.s_form ? (long long)s->pop_bytes : 0;
  return g;
}

bool uses_tile2d(const lbm_sim* s) {
  if (s->kernel == LBM_KERNEL_ROWS || !tile2d_eligible(s->params)) return false;
  return s->kernel == LBM_KERNEL_TILES || s->kernel == LBM_KERNEL_RESIDENT ||
         (long long)s->nx * s->ny <= SMALL_GRID_CELLS;
}

static int pitch_of(int nx) { return (nx + 31) / 32 * 32; }

static bool is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

static int check_params(int nx, int ny, const lbm_params* p) {
  if (!p) return set_error("params is NULL"), LBM_ERR_INVALID_ARG;
  if ((p->bc_x != LBM_PERIODIC && p->bc_x != LBM_WALL) || (p->bc_y != LBM_PERIODIC && p->bc_y != LBM_WALL))
    return set_error("bc_x/bc_y must be LBM_PERIODIC or LBM_WALL"), LBM_ERR_INVALID_ARG;
  if (nx < (p->bc_x == LBM_WALL ? 4 : 3) || ny < (p->bc_y == LBM_WALL ? 4 : 3))
    return set_error("grid %dx%d too small (>= 3, >= 4 along a walled axis)", nx, ny), LBM_ERR_INVALID_ARG;
  // byte offsets inside one population buffer are 32-bit (76 B per cell in FP32: 28 M cells)
  if ((long long)ny * pitch_of(nx) * state_bytes_per_cell(LBM_FP32) >= (1LL << 31))
    return set_error("grid %dx%d too large (one state buffer must stay below 2 GiB)", nx, ny), LBM_ERR_INVALID_ARG;
  if (!(p->tau_f > 0.5 && p->tau_g_A > 0.5 && p->tau_g_B > 0.5))
    return set_error("relaxation times must exceed 1/2"), LBM_ERR_INVALID_ARG;
  if (!(p->rho_A > 0 && p->rho_B > 0)) return set_error("densities must be positive"), LBM_ERR_INVALID_ARG;
  if (!(p->beta > 0 && p->kappa > 0 && p->phi_star > 0))
    return set_error("beta, kappa and phi_star must be positive"), LBM_ERR_INVALID_ARG;
  if (!(p->theta_M >= 0) || !(p->gravity == p->gravity))
    return set_error("theta_M must be >= 0 and gravity finite"), LBM_ERR_INVALID_ARG;
  if (p->storage != LBM_FP32 && p->storage != LBM_FP16_DEV && p->storage != LBM_BF16_DEV)
    return set_error("storage must be LBM_FP32, LBM_FP16_DEV or LBM_BF16_DEV"), LBM_ERR_INVALID_ARG;
  if (p->ch_conservative != 0 && p->ch_conservative != 1)
    return set_error("ch_conservative must be 0 or 1"), LBM_ERR_INVALID_ARG;
  if (p->fs_form != 0 && p->fs_form != 1) return set_error("fs_form must be 0 or 1"), LBM_ERR_INVALID_ARG;
  if (p->s_form != 0 && p->s_form != 1) return set_error("s_form must be 0 or 1"), LBM_ERR_INVALID_ARG;
  if (p->f_form != 0 && p->f_form != 1) return set_error("f_form must be 0 or 1"), LBM_ERR_INVALID_ARG;
  if (p->f_form && p->storage != LBM_FP32)
    return set_error("f_form 1 needs FP32 storage (its populations are O(phi))"), LBM_ERR_INVALID_ARG;
  return LBM_OK;
}

// Page-locked records, so that kernels write a simulation's diagnostics and its give-up word to the host and no copy
// follows.  One block for the process, allocated with the first simulation (allocating page-locked memory orders the
// streams of the device, so it is not done again); a simulation that finds no free record copies.
namespace {
class RecordPool {
 public:
  HostRecord* take() {
    std::lock_guard<std::mutex> lock(mu_);
    if (!tried_) {
      tried_ = true;
      void* p = nullptr;
      if (cudaHostAlloc(&p, SLOTS * sizeof(HostRecord), cudaHostAllocPortable) == cudaSuccess) {
        for (int k = SLOTS - 1; k >= 0; --k) free_[n_++] = static_cast<HostRecord*>(p) + k;
      } else {
        cudaGetLastError();
      }
    }
    if (n_ == 0) return nullptr;
    HostRecord* r = free_[--n_];
    r->gave_up = 0u;
    return r;
  }
  void give(HostRecord* d) {
    std::lock_guard<std::mutex> lock(mu_);
    free_[n_++] = d;
  }

 private:
  static constexpr int SLOTS = 512;
  std::mutex mu_;
  bool tried_ = false;
  int n_ = 0;
  HostRecord* free_[SLOTS];
};
RecordPool g_records;
}  // namespace

}  // namespace lbm

using namespace lbm;

extern "C" {

int lbm_params_from_sigma_W(double sigma, double W, double phi_star, double* beta, double* kappa) {
  if (!(sigma > 0 && W > 0 && phi_star > 0) || !beta || !kappa) {
    set_error("sigma, W and phi_star must be positive");
    return LBM_ERR_INVALID_ARG;
  }
  *kappa = 3.0 * sigma * W / (8.0 * phi_star * phi_star);
  *beta = 3.0 * sigma / (4.0 * W * phi_star * phi_star * phi_star * phi_star);
  return LBM_OK;
}

double lbm_tau_from_nu(double nu) { return 3.0 * nu + 0.5; }

size_t lbm_device_bytes(int nx, int ny, int storage) {
  const size_t plane = (size_t)ny * pitch_of(nx);
  return 2 * (size_t)state_bytes_per_cell(storage) * plane + N_FIELDS * plane * sizeof(float) +
         ((size_t)ny * DIAG_PARTIALS + 16) * sizeof(double);
}

size_t lbm_sim_device_bytes(const lbm_sim* s) {
  if (!s) return 0;
  return lbm_device_bytes(s->nx, s->ny, s->params.storage) + 2 * (s->buf_bytes - s->pop_bytes);
}

int lbm_create(int nx, int ny, const lbm_params* params, void* cuda_stream, lbm_sim** out) {
  Range range_("lbm_create");
  if (!out) return set_error("out is NULL"), LBM_ERR_INVALID_ARG;
  *out = nullptr;
  int rc = check_params(nx, ny, params);
  if (rc) return rc;
  lbm_sim* s = new (std::nothrow) lbm_sim();
  if (!s) return set_error("host allocation failed"), LBM_ERR_OOM;
  s->nx = nx;
  s->ny = ny;
  s->pitch = pitch_of(nx);
  s->plane = (long long)ny * s->pitch;
  s->params = *params;
  s->phys = make_phys(*params);
  s->phys2 = widen(s->phys);
  s->stream = (cudaStream_t)cuda_stream;
  const size_t pop_bytes = (size_t)state_bytes_per_cell(params->storage) * s->plane;
  s->pop_bytes = pop_bytes;
  s->buf_bytes = pop_bytes + (params->s_form ? 2 * sizeof(float) * (size_t)s->plane : 0);
  cudaError_t e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
    rc = cuda_fail(e, "lbm_create device query");
    delete s;
    return rc;
  }
  s->shape = march_shape(nx, ny, params->storage, params->s_form != 0, s->sms);
  const size_t field_bytes = (size_t)N_FIELDS * s->plane * sizeof(float);
  const size_t red_bytes = ((size_t)ny * DIAG_PARTIALS + 16) * sizeof(double);
  // Stream-ordered allocations from the device's memory pool, on the simulation's stream: unlike
  // cudaMalloc they do not order the other streams of the device, so a server can create a
  // simulation while others run.  The memory is ordered on s->stream (lbm_set_stream and
  // lbm_batch_add synchronise it before other streams use the state).
  if ((e = cudaMallocAsync(&s->buf[0], s->buf_bytes, s->stream)) != cudaSuccess ||
      (e = cudaMallocAsync(&s->buf[1], s->buf_bytes, s->stream)) != cudaSuccess ||
      (e = cudaMallocAsync(reinterpret_cast<void**>(&s->fields), field_bytes + red_bytes, s->stream)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&s->uploaded, cudaEventDisableTiming)) != cudaSuccess) {
    rc = cuda_fail(e, "lbm_create allocation");
    lbm_destroy(s);
    return rc;
  }
  // zero the pad columns once so no uninitialised memory is ever read back
  cudaMemsetAsync(s->buf[0], 0, s->buf_bytes, s->stream);
  cudaMemsetAsync(s->buf[1], 0, s->buf_bytes, s->stream);
  s->red = reinterpret_cast<double*>(s->fields + (size_t)N_FIELDS * s->plane);   // behind the work planes
  cudaMemsetAsync(s->fields, 0, field_bytes + red_bytes, s->stream);
  if ((e = cudaGetLastError()) != cudaSuccess) {
    rc = cuda_fail(e, "lbm_create memset");
    lbm_destroy(s);
    return rc;
  }
  s->slot = g_records.take();
  *out = s;
  return LBM_OK;
}

// One nx*ny field between a pitched work plane and a caller's packed buffer.  When the pitch
// equals nx both are one contiguous block, copied as such rather than row by row.
static cudaError_t copy_field(const lbm_sim* s, float* dst, size_t dpitch, const float* src, size_t spitch,
                              cudaMemcpyKind kind) {
  const size_t row = (size_t)s->nx * sizeof(float);
  if (dpitch == row && spitch == row)
    return cudaMemcpyAsync(dst, src, row * s->ny, kind, s->stream);
  return cudaMemcpy2DAsync(dst, dpitch, src, spitch, row, s->ny, kind, s->stream);
}

// A new state re-arms the resident kernel's waits: a launch that gave up is forgotten.
static cudaError_t rearm_resident(lbm_sim* s) {
  s->res_used = false;
  return resident_reset(s);
}

// Device memory that this simulation's kernels can address as floats: on the current device or managed, and aligned.
static bool addressable(const void* p) {
  cudaPointerAttributes a;
  int dev = 0;
  if (reinterpret_cast<uintptr_t>(p) % sizeof(float) != 0) return false;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev);
}

// Initial field k (0 phi0, 1 ux0, 2 uy0, 3 p0): read in place by the initialisation kernel where it can address the
// memory (copying device fields into work planes first took a third of its traffic), else through its work plane.
static int take_field(lbm_sim* s, int k, const float* src, InitIn* in, bool* host) {
  in->f[k] = src;
  in->pitch[k] = s->nx;
  if (!src || addressable(src)) return LBM_OK;
  const int plane = k == 0 ? 0 : k + 1;
  float* dst = s->fields + (long long)plane * s->plane;
  const bool dev = is_device_ptr(src);
  const cudaError_t e = copy_field(s, dst, (size_t)s->pitch * sizeof(float), src, (size_t)s->nx * sizeof(float),
                                   dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_init_fields upload");
  in->f[k] = dst;
  in->pitch[k] = s->pitch;
  *host = *host || !dev;
  return LBM_OK;
}

int lbm_init_fields(lbm_sim* s, const float* phi0, const float* ux0, const float* uy0, const float* p0) {
  Range range_("lbm_init_fields");
  if (!s || !phi0) return set_error("sim and phi0 are required"), LBM_ERR_INVALID_ARG;
  int rc;
  InitIn in{};
  bool host_input = false;
  if ((rc = take_field(s, 0, phi0, &in, &host_input)) || (rc = take_field(s, 1, ux0, &in, &host_input)) ||
      (rc = take_field(s, 2, uy0, &in, &host_input)) || (rc = take_field(s, 3, p0, &in, &host_input)))
    return rc;
  cudaError_t e = cudaSuccess;
  if (host_input && (e = cudaEventRecord(s->uploaded, s->stream)) != cudaSuccess) return cuda_fail(e, "lbm_init_fields record");
  e = launch_init(s, in, s->stream);
  if (e == cudaSuccess) e = rearm_resident(s);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_init_fields launch");
  s->launches += s->params.s_form ? 2 : 1;
  s->steps = 0;
  // host inputs must be consumed before return (pageable copies already are; pinned ones not):
  // wait for the copies only, so the initialisation kernels overlap the caller's next launches.
  // Any one host input is enough to wait: phi0 may be on the device while ux0 is pinned.
  if (host_input && (e = cudaEventSynchronize(s->uploaded)) != cudaSuccess)
    return cuda_fail(e, "lbm_init_fields sync");
  return LBM_OK;
}

// nplanes consecutive nx*ny fields between consecutive pitched work planes (starting at plane
// k0) and a caller's packed block: one copy (one 2D copy when the pitch differs from nx).
static cudaError_t copy_planes(const lbm_sim* s, int k0, int nplanes, float* packed, bool to_work,
                               cudaMemcpyKind kind) {
  float* work = s->fields + (long long)k0 * s->plane;
  const size_t row = (size_t)s->nx * sizeof(float), wpitch = (size_t)s->pitch * sizeof(float);
  const size_t rows = (size_t)nplanes * s->ny;   // consecutive work planes are ny pitched rows apart
  if (wpitch == row) {
    return to_work ? cudaMemcpyAsync(work, packed, row * rows, kind, s->stream)
                   : cudaMemcpyAsync(packed, work, row * rows, kind, s->stream);
  }
  return to_work ? cudaMemcpy2DAsync(work, wpitch, packed, row, row, rows, kind, s->stream)
                 : cudaMemcpy2DAsync(packed, row, work, wpitch, row, rows, kind, s->stream);
}

int lbm_init_fields_packed(lbm_sim* s, const float* fields) {
  Range range_("lbm_init_fields_packed");
  if (!s || !fields) return set_error("sim and fields are required"), LBM_ERR_INVALID_ARG;
  const size_t n = (size_t)s->nx * s->ny;
  InitIn in{};
  bool host = false;
  cudaError_t e = cudaSuccess;
  if (addressable(fields)) {
    for (int k = 0; k < 4; ++k) {
      in.f[k] = fields + k * n;
      in.pitch[k] = s->nx;
    }
  } else {
    host = !is_device_ptr(fields);
    const cudaMemcpyKind kind = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    // one copy into consecutive work planes
    e = copy_planes(s, 0, 4, const_cast<float*>(fields), true, kind);   // (read only)
    if (e == cudaSuccess && host) e = cudaEventRecord(s->uploaded, s->stream);
    if (e != cudaSuccess) return cuda_fail(e, "lbm_init_fields_packed upload");
    for (int k = 0; k < 4; ++k) {
      in.f[k] = s->fields + (long long)k * s->plane;
      in.pitch[k] = s->pitch;
    }
  }
  e = launch_init(s, in, s->stream);
  if (e == cudaSuccess) e = rearm_resident(s);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_init_fields_packed launch");
  s->launches += s->params.s_form ? 2 : 1;
  s->steps = 0;
  if (host && (e = cudaEventSynchronize(s->uploaded)) != cudaSuccess)
    return cuda_fail(e, "lbm_init_fields_packed sync");
  return LBM_OK;
}

// Zero the row march's give-up words, on a stream that has been synchronised (both or neither are raised).
static cudaError_t clear_gave_up(lbm_sim* s) {
  if (s->slot) {
    volatile unsigned int& host = s->slot->gave_up;
    if (host == 0u) return cudaSuccess;
    host = 0u;
  }
  return cudaMemsetAsync(gave_up(s), 0, sizeof(unsigned int), s->stream);
}

// Behind a synchronisation of the stream: LBM_ERR_TIMEOUT if a wait of the row march ran out since the state was set or
// this was last read.  Costs a look at page-locked memory (a copy for a simulation without a record).
static int march_status(lbm_sim* s) {
  unsigned int st = 0;
  cudaError_t e = cudaSuccess;
  if (s->slot) {
    st = *static_cast<volatile unsigned int*>(&s->slot->gave_up);
  } else {
    e = cudaMemcpyAsync(&st, gave_up(s), sizeof st, cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(e, "status copy");
  }
  if (st == 0) return LBM_OK;
  if ((e = clear_gave_up(s)) != cudaSuccess) return cuda_fail(e, "status reset");
  set_error("a wait of the row march ran out (%lld ns); the state is undefined", s->wait_ns);
  return LBM_ERR_TIMEOUT;
}

// Status of the launches since the last read; synchronises the stream.  A launch that gave up returns LBM_ERR_TIMEOUT
// and re-arms the waits (flags and status zeroed).
static int read_status(lbm_sim* s) {
  unsigned int st = 0;
  cudaError_t e = cudaSuccess;
  if (s->res_used)
    e = cudaMemcpyAsync(&st, s->res_mem + resident_tiles(s->nx, s->ny), sizeof st, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "status");
  s->res_used = false;
  if (st == 0) return march_status(s);
  if ((e = resident_reset(s)) != cudaSuccess) return cuda_fail(e, "status reset");
  set_error("a wait of the resident step kernel ran out (%lld ns); the state is undefined", s->wait_ns);
  return LBM_ERR_TIMEOUT;
}

int lbm_step(lbm_sim* s, int n) {
  Range range_("lbm_step");
  if (!s || n < 0) return set_error("invalid sim or step count"), LBM_ERR_INVALID_ARG;
  if (s->batch) return set_error("simulation is a batch member; step it through its batch"), LBM_ERR_INVALID_ARG;
  if (n >= 2 && s->kernel == LBM_KERNEL_RESIDENT) {
    Grid g = make_grid(s, s->buf[s->cur], s->buf[s->cur ^ 1]);
    cudaError_t e = launch_resident(s, g, n);
    if (e != cudaSuccess) return cuda_fail(e, "lbm_step resident launch");
    s->cur ^= n & 1;
    s->steps += n;
    s->launches++;
    return LBM_OK;
  }
  const bool tiles = uses_tile2d(s);
  for (int i = 0; i < n; ++i) {
    Grid g = make_grid(s, s->buf[s->cur], s->buf[s->cur ^ 1]);
    g.wait_hold = s->hold;
    cudaError_t e = tiles ? launch_tile2d(s->phys, g, nullptr, s->sms, s->stream) : launch_step(s->phys2, g, s->stream);
    if (e != cudaSuccess) return cuda_fail(e, "lbm_step launch");
    s->cur ^= 1;
    s->steps++;
    s->launches++;
  }
  return LBM_OK;
}

// The moment pass of the current state.  Small grids take the tile kernel's three passes, whose
// latency is that of one tile, instead of a march over rows.
static cudaError_t moments_of(const lbm_sim* s, const Grid& g, const MomentOut& mo) {
  if (s->params.s_form == 0 && (long long)s->nx * s->ny <= SMALL_GRID_MOMENTS)
    return launch_tile2d(s->phys, g, &mo, s->sms, s->stream);
  return launch_moments(s->phys2, g, mo, s->stream);
}

static int compute_moments(lbm_sim* s) {
  Grid g = make_grid(s, s->buf[s->cur], nullptr);
  MomentOut mo{s->fields, s->fields + s->plane, s->fields + 2 * s->plane, s->fields + 3 * s->plane,
               s->fields + 4 * s->plane, nullptr, nullptr, s->pitch};
  cudaError_t e = moments_of(s, g, mo);
  if (e != cudaSuccess) return cuda_fail(e, "moments launch");
  s->launches++;
  return LBM_OK;
}

// Copy fields planes 0..n-1 (pitched) into the caller's nx*ny outputs (null ones skipped), then
// synchronise the stream.
static int copy_out(lbm_sim* s, float* const* outs, int n, const char* what) {
  for (int k = 0; k < n; ++k) {
    if (!outs[k]) continue;
    const cudaMemcpyKind kind = is_device_ptr(outs[k]) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    cudaError_t e = copy_field(s, outs[k], (size_t)s->nx * sizeof(float), s->fields + (long long)k * s->plane,
                               (size_t)s->pitch * sizeof(float), kind);
    if (e != cudaSuccess) return cuda_fail(e, what);
  }
  cudaError_t e = cudaStreamSynchronize(s->stream);
  return e == cudaSuccess ? march_status(s) : cuda_fail(e, what);
}

// Outputs of the moment pass.  Where it can address all of a call's outputs it writes them in place; otherwise all go
// through the work planes and are copied.  Page-locked host memory is also addressable by the kernel, but its 4-byte
// stores across NVLink-C2C ran slower than the bulk copy (c3 end to end: 11.76 against 12.1 GLUPS), so host
// outputs are always copied.
static bool all_direct(float* const* outs, int n) {
  for (int k = 0; k < n; ++k)
    if (outs[k] && !addressable(outs[k])) return false;
  return true;
}

int lbm_moments(lbm_sim* s, float* phi, float* rho, float* ux, float* uy, float* p) {
  Range range_("lbm_moments");
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  float* outs[5] = {phi, rho, ux, uy, p};
  float* dst[5];
  // in place: all outputs, or, where the work planes have the same pitch, those that can be
  const bool direct = all_direct(outs, 5);
  float* staged[5] = {};
  for (int k = 0; k < 5; ++k) {
    dst[k] = outs[k];
    if (!outs[k] || direct || (s->pitch == s->nx && addressable(outs[k]))) continue;
    dst[k] = s->fields + (long long)k * s->plane;
    staged[k] = outs[k];
  }
  Grid g = make_grid(s, s->buf[s->cur], nullptr);
  MomentOut mo{dst[0], dst[1], dst[2], dst[3], dst[4], nullptr, nullptr, direct ? s->nx : s->pitch};
  cudaError_t e = moments_of(s, g, mo);
  if (e != cudaSuccess) return cuda_fail(e, "moments launch");
  s->launches++;
  return copy_out(s, staged, 5, "lbm_moments copy");
}

int lbm_moments_packed(lbm_sim* s, float* fields) {
  Range range_("lbm_moments_packed");
  if (!s || !fields) return set_error("sim and fields are required"), LBM_ERR_INVALID_ARG;
  const bool direct = addressable(fields);
  float* dst = direct ? fields : s->fields;
  const size_t stride = direct ? (size_t)s->nx * s->ny : (size_t)s->plane;
  Grid g = make_grid(s, s->buf[s->cur], nullptr);
  MomentOut mo{dst, dst + stride, dst + 2 * stride, dst + 3 * stride, dst + 4 * stride, nullptr, nullptr, direct ? s->nx : s->pitch};
  cudaError_t e = moments_of(s, g, mo);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_moments_packed launch");
  s->launches++;
  if (!direct) {
    const cudaMemcpyKind kind = is_device_ptr(fields) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    e = copy_planes(s, 0, 5, fields, false, kind);
    if (e != cudaSuccess) return cuda_fail(e, "lbm_moments_packed copy");
  }
  e = cudaStreamSynchronize(s->stream);
  return e == cudaSuccess ? march_status(s) : cuda_fail(e, "lbm_moments_packed sync");
}

int lbm_interfacial_force(lbm_sim* s, float* fa_x, float* fa_y) {
  Range range_("lbm_interfacial_force");
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  Grid g = make_grid(s, s->buf[s->cur], nullptr);
  float* outs[2] = {fa_x, fa_y};
  MomentOut mo{};
  const bool direct = fa_x && fa_y && all_direct(outs, 2);   // the kernel writes both components
  mo.fax = direct ? fa_x : s->fields;
  mo.fay = direct ? fa_y : s->fields + s->plane;
  mo.pitch = direct ? s->nx : s->pitch;
  cudaError_t e = moments_of(s, g, mo);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_interfacial_force launch");
  s->launches++;
  return copy_out(s, outs, direct ? 0 : 2, "lbm_interfacial_force copy");
}

int lbm_diagnostics(lbm_sim* s, lbm_diag* out) {
  Range range_("lbm_diagnostics");
  if (!s || !out) return set_error("sim and out are required"), LBM_ERR_INVALID_ARG;
  int rc = compute_moments(s);
  if (rc) return rc;
  cudaError_t e = launch_diag(s, s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "diagnostics launch");
  s->launches++;
  if (!s->slot) {
    e = cudaMemcpyAsync(&s->h_diag, s->red + (long long)s->ny * DIAG_PARTIALS, sizeof(lbm_diag), cudaMemcpyDeviceToHost,
                        s->stream);
    if (e != cudaSuccess) return cuda_fail(e, "diagnostics copy");
  }
  if ((rc = read_status(s)) != LBM_OK) return rc;
  *out = s->slot ? s->slot->diag : s->h_diag;
  if (!out->finite) {
    set_error("simulation diverged (non-finite state) at step %lld", out->step);
    return LBM_ERR_DIVERGED;
  }
  return LBM_OK;
}

int lbm_destroy(lbm_sim* s) {
  if (!s) return LBM_OK;
  if (s->stream || s->buf[0]) cudaStreamSynchronize(s->stream);
  // back to the pool, ordered on the stream: no device-wide synchronisation
  for (void* p : {s->buf[0], s->buf[1], static_cast<void*>(s->fields), static_cast<void*>(s->res_mem)})
    if (p) cudaFreeAsync(p, s->stream);
  if (s->uploaded) cudaEventDestroy(s->uploaded);
  if (s->slot) g_records.give(s->slot);
  delete s;
  return LBM_OK;
}

long long lbm_step_count(const lbm_sim* s) { return s ? s->steps : -1; }

}  // extern "C"

namespace {
struct CkptHeader {
  uint32_t magic;       // "LBMC"
  uint32_t version;     // 2: blocked population layout (32-cell blocks)
  int32_t nx, ny, pitch, storage;
  int64_t steps;
  uint64_t payload;     // bytes of the population buffer that follows
  uint64_t reserved[3];
};
static_assert(sizeof(CkptHeader) == 64, "checkpoint header is 64 bytes");
constexpr uint32_t CKPT_MAGIC = 0x434d424cu;   // "LBMC" little-endian
constexpr uint32_t CKPT_VERSION = 2;

size_t payload_bytes(const lbm_sim* s) { return s->buf_bytes; }

// The current state between its buffer and a checkpoint's payload (blocks of 32 cells, then the s_form planes).  A
// payload in memory that this device addresses is read or written by the reordering kernel itself; otherwise (host
// memory, another device's) the populations pass through the field work planes and the diagnostics' partials behind
// them, as many at a time as those hold (no allocation: a server evicts when memory is short; and not through the other
// state buffer, whose pad columns would not keep what they hold).
cudaError_t move_payload(lbm_sim* s, char* payload, bool to_payload, bool dev) {
  char* state = static_cast<char*>(s->buf[s->cur]);
  const long long groups = reorder_groups(s, to_payload);
  cudaError_t e = cudaSuccess;
  if (addressable(payload)) {
    e = launch_reorder(s, state, payload, 0, groups, to_payload, s->stream);
  } else {
    const cudaMemcpyKind kind = dev ? cudaMemcpyDeviceToDevice : (to_payload ? cudaMemcpyDeviceToHost : cudaMemcpyHostToDevice);
    const long long room = reorder_fit(s, to_payload, N_FIELDS * (size_t)s->plane * sizeof(float) + (size_t)s->ny * DIAG_PARTIALS * sizeof(double));
    for (long long k = 0; k < groups && e == cudaSuccess; k += room) {
      const long long end = std::min(groups, k + room), at = reorder_offset(s, to_payload, k);
      const size_t n = (size_t)((end < groups ? reorder_offset(s, to_payload, end) : (long long)s->pop_bytes) - at);
      if (to_payload) {
        e = launch_reorder(s, state, s->fields, k, end, true, s->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(payload + at, s->fields, n, kind, s->stream);
      } else {
        e = cudaMemcpyAsync(s->fields, payload + at, n, kind, s->stream);
        if (e == cudaSuccess) e = launch_reorder(s, state, s->fields, k, end, false, s->stream);
      }
    }
  }
  const size_t rest = s->buf_bytes - s->pop_bytes;
  if (e == cudaSuccess && rest) {
    char *planes = state + s->pop_bytes, *part = payload + s->pop_bytes;
    e = to_payload ? cudaMemcpyAsync(part, planes, rest, dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s->stream)
                   : cudaMemcpyAsync(planes, part, rest, dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s->stream);
  }
  return e;
}
}  // namespace

extern "C" {

size_t lbm_checkpoint_bytes(const lbm_sim* s) { return s ? sizeof(CkptHeader) + payload_bytes(s) : 0; }

int lbm_checkpoint(lbm_sim* s, void* buf, size_t bytes) {
  Range range_("lbm_checkpoint");
  if (!s || !buf) return set_error("sim and buf are required"), LBM_ERR_INVALID_ARG;
  if (s->batch) return set_error("remove the simulation from its batch before a checkpoint"), LBM_ERR_INVALID_ARG;
  if (bytes < lbm_checkpoint_bytes(s))
    return set_error("checkpoint buffer of %zu bytes, %zu needed", bytes, lbm_checkpoint_bytes(s)), LBM_ERR_INVALID_ARG;
  CkptHeader h{};
  h.magic = CKPT_MAGIC;
  h.version = CKPT_VERSION;
  h.nx = s->nx;
  h.ny = s->ny;
  h.pitch = s->pitch;
  h.storage = s->params.storage;
  h.steps = s->steps;
  h.payload = payload_bytes(s);
  const bool dev = is_device_ptr(buf);
  cudaError_t e = dev ? cudaMemcpyAsync(buf, &h, sizeof(h), cudaMemcpyHostToDevice, s->stream) : cudaSuccess;
  if (e == cudaSuccess)
    e = move_payload(s, static_cast<char*>(buf) + sizeof(h), true, dev);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);   // h lives on this stack frame
  if (e == cudaSuccess && !dev) memcpy(buf, &h, sizeof(h));     // (behind the stream's earlier work on buf)
  return e == cudaSuccess ? march_status(s) : cuda_fail(e, "lbm_checkpoint copy");
}

int lbm_restore(lbm_sim* s, const void* buf, size_t bytes) {
  Range range_("lbm_restore");
  if (!s || !buf) return set_error("sim and buf are required"), LBM_ERR_INVALID_ARG;
  if (s->batch) return set_error("remove the simulation from its batch before a restore"), LBM_ERR_INVALID_ARG;
  if (bytes < sizeof(CkptHeader)) return set_error("checkpoint shorter than its header"), LBM_ERR_INVALID_ARG;
  const bool dev = is_device_ptr(buf);
  CkptHeader h{};
  cudaError_t e = dev ? cudaMemcpyAsync(&h, buf, sizeof(h), cudaMemcpyDeviceToHost, s->stream) : cudaSuccess;
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e == cudaSuccess && !dev) memcpy(&h, buf, sizeof(h));
  if (e != cudaSuccess) return cuda_fail(e, "lbm_restore header");
  if (h.magic != CKPT_MAGIC || h.version != CKPT_VERSION) return set_error("not a checkpoint (bad magic or version)"), LBM_ERR_INVALID_ARG;
  if (h.nx != s->nx || h.ny != s->ny || h.pitch != s->pitch || h.storage != s->params.storage ||
      h.payload != payload_bytes(s))
    return set_error("checkpoint of a %dx%d storage-%d grid, simulation is %dx%d storage %d", h.nx, h.ny, h.storage,
                     s->nx, s->ny, s->params.storage), LBM_ERR_INVALID_ARG;
  if (bytes < sizeof(h) + h.payload) return set_error("checkpoint truncated"), LBM_ERR_INVALID_ARG;
  e = move_payload(s, const_cast<char*>(static_cast<const char*>(buf)) + sizeof(h), false, dev);
  if (e == cudaSuccess) e = rearm_resident(s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e == cudaSuccess) e = clear_gave_up(s);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_restore copy");
  s->steps = h.steps;
  return LBM_OK;
}

int lbm_set_stream(lbm_sim* s, void* stream) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  // the state's allocation and earlier work are ordered on the old stream
  cudaError_t e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "lbm_set_stream sync");
  s->stream = (cudaStream_t)stream;
  return LBM_OK;
}

int lbm_set_tile(lbm_sim* s, int threads, int seg_rows) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  if (threads && threads != 64 && threads != 128 && threads != 256)
    return set_error("threads must be 64, 128 or 256"), LBM_ERR_INVALID_ARG;
  if (seg_rows < 0) return set_error("seg_rows must be >= 1"), LBM_ERR_INVALID_ARG;
  if (seg_rows) s->seg_h = seg_rows;
  return LBM_OK;
}

int lbm_set_tile_auto(lbm_sim* s) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  s->seg_h = 0;
  return LBM_OK;
}

int lbm_set_kernel(lbm_sim* s, int kernel) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  if (kernel != LBM_KERNEL_AUTO && kernel != LBM_KERNEL_ROWS && kernel != LBM_KERNEL_TILES &&
      kernel != LBM_KERNEL_RESIDENT)
    return set_error("kernel must be LBM_KERNEL_AUTO, _ROWS, _TILES or _RESIDENT"), LBM_ERR_INVALID_ARG;
  if ((kernel == LBM_KERNEL_TILES || kernel == LBM_KERNEL_RESIDENT) && !tile2d_eligible(s->params))
    return set_error("the tile kernels need s_form 0 and f_form 0"), LBM_ERR_INVALID_ARG;
  s->kernel = kernel;
  return LBM_OK;
}

int lbm_set_wait_limit(lbm_sim* s, long long timeout_ns, int hold_tile) {
  if (!s || timeout_ns <= 0) return set_error("invalid sim or timeout"), LBM_ERR_INVALID_ARG;
  s->wait_ns = timeout_ns;
  s->hold = hold_tile < 0 ? -1 : hold_tile;
  return LBM_OK;
}

int lbm_step_status(lbm_sim* s) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  return read_status(s);
}

int lbm_active_kernel(const lbm_sim* s) {
  if (!s) return set_error("sim is NULL"), LBM_ERR_INVALID_ARG;
  if (s->kernel == LBM_KERNEL_RESIDENT) return LBM_KERNEL_RESIDENT;
  return uses_tile2d(s) ? LBM_KERNEL_TILES : LBM_KERNEL_ROWS;
}

long long lbm_launch_count(const lbm_sim* s) { return s ? s->launches : -1; }

const char* lbm_strerror(int code) {
  switch (code) {
    case LBM_OK: return "ok";
    case LBM_ERR_INVALID_ARG: return "invalid argument";
    case LBM_ERR_OOM: return "out of device memory";
    case LBM_ERR_BUDGET: return "device-memory budget exceeded";
    case LBM_ERR_DIVERGED: return "simulation diverged";
    case LBM_ERR_TIMEOUT: return "timed out";
    case LBM_ERR_CUDA: return "CUDA error";
    default: return "unknown error";
  }
}

const char* lbm_last_error(void) { return g_last_error.c_str(); }

}  // extern "C"
