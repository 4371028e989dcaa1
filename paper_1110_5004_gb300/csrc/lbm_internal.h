// Host-side internals shared by the translation units of liblbm (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <string>

#include <nvtx3/nvToolsExt.h>  // header-only; a no-op unless a profiler is attached

#include "lbm.h"  // include/ is on the include path
#include "lbm_device.cuh"

namespace lbm {
constexpr long long WAIT_TRY_NS = 1300;   // what a try of a row march's wait takes (measured: 26 ms for 20 003)
constexpr long long WAIT_LEAST_NS = 1000000;   // its least limit: longer than copies take on a busy device
// Page-locked words of a simulation that its kernels write: the host reads them without a copy.
struct HostRecord {
  lbm_diag diag;
  unsigned int gave_up;
};
}  // namespace lbm

namespace lbm {
// Threads per CTA of the row march, strips across the grid and columns per lane.
struct MarchShape {
  int nt = 0, strips = 0, width = 0;
};
}  // namespace lbm

struct lbm_sim {
  int nx = 0, ny = 0, pitch = 0;
  long long plane = 0;      // elements per plane
  lbm_params params{};
  lbm::Phys phys{};
  lbm::Phys2 phys2{};       // the same, each constant doubled
  cudaStream_t stream = nullptr;
  void* buf[2] = {nullptr, nullptr};   // post-collision state, buf_bytes each
  size_t buf_bytes = 0;                // populations (+ rho, div(rho u) planes with s_form = 1)
  size_t pop_bytes = 0;                // populations only
  int cur = 0;                         // buffer holding the current state
  float* fields = nullptr;             // 6 planes: phi, rho, ux, uy, p, mu (moments and init)
  double* red = nullptr;               // reduction scratch: ny rows x 12 partials + final record
  lbm_diag h_diag{};                   // host copy of the final record, for a simulation without a slot
  lbm::HostRecord* slot = nullptr;     // or null (more simulations than records)
  cudaEvent_t uploaded = nullptr;      // recorded after lbm_init_fields' host-to-device copies
  long long steps = 0;
  long long launches = 0;
  int kernel = LBM_KERNEL_AUTO;        // step kernel choice (lbm_set_kernel)
  lbm::MarchShape shape;               // of the row march
  int seg_h = 0;                       // rows per CTA (0: one wave of resident CTAs)
  int sms = 0;                         // multiprocessors of the device
  // resident tile kernel (lbm_tile2d.cu): per-tile step flags, the status word and the reach
  // table in one stream-ordered allocation made at first use
  unsigned int* res_mem = nullptr;
  unsigned int res_base = 0;           // flag value of every tile between launches
  long long wait_ns = 1000000000LL;    // limit of a wait, of the resident kernel and of the row march
  int hold = -1;                       // test hook: this tile never announces a finished step, or gets its rows
  bool res_used = false;               // a resident launch ran since the status was last read
  lbm_batch* batch = nullptr;
};

namespace lbm {

// Named range on the profiler's timeline for the duration of one entry point.
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
  Range(const Range&) = delete;
  Range& operator=(const Range&) = delete;
};

constexpr int N_FIELDS = 6;
constexpr int DIAG_PARTIALS = 12;
// Words in the spare doubles behind the diagnostics record: raised by a wait of the row march that ran out
// (GiveUp::word); blocks of a diagnostics launch that have finished.
inline unsigned int* gave_up(const lbm_sim* s) { return reinterpret_cast<unsigned int*>(s->red + (size_t)s->ny * DIAG_PARTIALS + 14); }
inline unsigned int* diag_done(const lbm_sim* s) { return gave_up(s) + 1; }

void set_error(const char* fmt, ...);
int cuda_fail(cudaError_t e, const char* what);
Phys make_phys(const lbm_params& p);
Grid make_grid(const lbm_sim* s, const void* src, void* dst);
// The fewest strips of two lanes, all alike, in which CTAs of nt threads can march nx columns; strips = 0: none.
MarchShape march_shape_of(int nx, int storage, bool sd, int nt);
// The best of the thread counts.
MarchShape march_shape(int nx, int ny, int storage, bool sd, int sms);
// The row march's part of a grid; seg_h = 0 picks the segment height that puts about one full wave of CTAs on `sms`
// multiprocessors.
void tile_geometry(const MarchShape& m, int seg_h, int sms, Grid* g);
// The small-grid step kernel (lbm_tile2d.cu): s_form 0 and f_form 0.
bool tile2d_eligible(const lbm_params& p);
// 384-thread CTAs when the grid's tiles fit one wave of them on `sms` multiprocessors, else 256.
// mo: null for a step, else the moment pass into it.
cudaError_t launch_tile2d(const Phys& P, const Grid& g, const MomentOut* mo, int sms, cudaStream_t st);
// Grids of at most this many cells take the tile kernel for their moments (one call, kernel and host: 128^2
// 18.5 us against 21.1 for the row march, 256 x 1024 27.6 against 29.1; 700^2 49.4 against 42.9).
constexpr long long SMALL_GRID_MOMENTS = 1 << 18;
// Shared memory to ask for so that at most `cap` CTAs fit on an SM, at least `need` (`need` where the device's limits
// cannot be read).
int smem_for_cap(int need, int cap);
// Grids of at most this many cells run the small-grid kernel by default (measured faster up to
// 2^18 cells, slower from 2^19 on, with and without x walls).
constexpr long long SMALL_GRID_CELLS = 1 << 18;
bool uses_tile2d(const lbm_sim* s);
// The resident form: one launch of n >= 2 steps (flags and reach table prepared on first use).
int resident_tiles(int nx, int ny);
cudaError_t resident_prepare(lbm_sim* s);
cudaError_t resident_reset(lbm_sim* s);
cudaError_t launch_resident(lbm_sim* s, const Grid& g, int n);

// launchers (return cudaError_t of the launch)
cudaError_t launch_step(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_step_fp32(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_step_fp16(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_step_bf16(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_narrow_fp32(const Phys2& P, const Grid& g, cudaStream_t st);   // 64 and 32 threads
cudaError_t launch_narrow_fp16(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_narrow_bf16(const Phys2& P, const Grid& g, cudaStream_t st);
cudaError_t launch_moments(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st);
cudaError_t launch_moments_narrow(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st);
cudaError_t launch_init(const lbm_sim* s, const InitIn& in, cudaStream_t st);
// Groups of blocks in which populations move between a state buffer and a checkpoint's order: how many the grid has, at
// what byte of the order a group starts, how many fit into `bytes` (at least one into a simulation's work planes and
// partials), and the move of [k0, k1), `lin` (4-byte aligned) being the place of group k0.
long long reorder_groups(const lbm_sim* s, bool out);
long long reorder_offset(const lbm_sim* s, bool out, long long k);
long long reorder_fit(const lbm_sim* s, bool out, size_t bytes);
cudaError_t launch_reorder(const lbm_sim* s, void* state, void* lin, long long k0, long long k1, bool out, cudaStream_t st);
cudaError_t launch_diag(const lbm_sim* s, cudaStream_t st);  // from fields -> red -> final record

}  // namespace lbm
