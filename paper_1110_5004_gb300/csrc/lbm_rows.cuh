// The row-march kernel of one simulation and its launch.  The storages and the moment pass are
// compiled in translation units of their own (lbm_rows_fp32.cu, ...), so that the build runs them in parallel.
#pragma once
#include "lbm_internal.h"
#include "lbm_march.cuh"

namespace lbm {

// Two CTAs of 128 threads per SM: shared memory (113 KB each in FP32 storage) and up to 255 registers; or 4 of 64, 8 of 32.
template <int MODE, int ST, bool SD, bool FF, bool XW, int NT>
__global__ void __launch_bounds__(NT, march_ctas(NT)) k_march(const __grid_constant__ Phys2 P, const __grid_constant__ Grid g,
                                                       const __grid_constant__ MomentOut mo) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  MarchSmem<ST, SD, NT>& sm = *reinterpret_cast<MarchSmem<ST, SD, NT>*>(smem_raw);
  march_init(sm);
  StageAt fat, gat;
  march<MODE, ST, SD, FF, XW, true, NT>(P, g, &g.give_up, mo, blockIdx.x % g.n_strips, blockIdx.x / g.n_strips, sm, fat, gat);
}

template <int MODE, int ST, bool SD, bool FF, bool XW, int NT>
static cudaError_t launch_march(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  static_assert((sizeof(MarchSmem<ST, SD, NT>) + 1024) * march_ctas(NT) <= 233472, "the CTAs of an SM fit its shared memory");
  // set once, thread-safely (host threads may step simulations concurrently; one GPU per process)
  static const cudaError_t attr_set = cudaFuncSetAttribute(
      k_march<MODE, ST, SD, FF, XW, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MarchSmem<ST, SD, NT>));
  if (attr_set != cudaSuccess) return attr_set;
  const int tiles = g.n_strips * ((g.ny + g.seg_h - 1) / g.seg_h);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = sizeof(MarchSmem<ST, SD, NT>);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // consecutive steps overlap their launches
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_march<MODE, ST, SD, FF, XW, NT>, P, g, mo);
}

template <int MODE, int ST, bool SD, bool FF, int NT>
static cudaError_t launch_rows_xw(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  return g.bc_x == BC_WALL ? launch_march<MODE, ST, SD, FF, true, NT>(P, g, mo, st)
                           : launch_march<MODE, ST, SD, FF, false, NT>(P, g, mo, st);
}

template <int MODE, int ST, int NT>
static cudaError_t launch_rows_nt(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  // the forced order-parameter form changes only the step's f collision (FP32 storage only)
  if constexpr (MODE == MODE_STEP && ST == ST_FP32) {
    if (P.f_forced)
      return P.s_direct ? launch_rows_xw<MODE, ST, true, true, NT>(P, g, mo, st) : launch_rows_xw<MODE, ST, false, true, NT>(P, g, mo, st);
  }
  return P.s_direct ? launch_rows_xw<MODE, ST, true, false, NT>(P, g, mo, st) : launch_rows_xw<MODE, ST, false, false, NT>(P, g, mo, st);
}

template <int MODE, int ST>
static cudaError_t launch_rows_narrow(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  return g.march_nt == 64 ? launch_rows_nt<MODE, ST, 64>(P, g, mo, st) : launch_rows_nt<MODE, ST, 32>(P, g, mo, st);
}

}  // namespace lbm
