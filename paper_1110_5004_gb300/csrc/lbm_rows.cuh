// The row-march kernel of one simulation and its launch.  The storages and the moment pass are
// compiled in translation units of their own (lbm_rows_fp32.cu, ...), so that the build runs them in parallel.
#pragma once
#include "lbm_internal.h"
#include "lbm_march.cuh"

namespace lbm {

// Two CTAs of 128 threads per SM: shared memory (113 KB each in FP32 storage) and up to 255 registers.
template <int MODE, int ST, bool SD, bool FF, bool XW>
__global__ void __launch_bounds__(MARCH_NT, MARCH_CTAS) k_march(const __grid_constant__ Phys2 P, const __grid_constant__ Grid g,
                                                       const __grid_constant__ MomentOut mo) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  MarchSmem<ST, SD>& sm = *reinterpret_cast<MarchSmem<ST, SD>*>(smem_raw);
  march_init(sm);
  StageAt fat, gat;
  march<MODE, ST, SD, FF, XW, true>(P, g, &g.wait, mo, blockIdx.x % g.n_strips, blockIdx.x / g.n_strips, sm, fat, gat);
}

template <int MODE, int ST, bool SD, bool FF, bool XW>
static cudaError_t launch_march(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  // set once, thread-safely (host threads may step simulations concurrently; one GPU per process)
  static const cudaError_t attr_set = cudaFuncSetAttribute(
      k_march<MODE, ST, SD, FF, XW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MarchSmem<ST, SD>));
  if (attr_set != cudaSuccess) return attr_set;
  const int tiles = g.n_strips * ((g.ny + g.seg_h - 1) / g.seg_h);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles);
  cfg.blockDim = dim3(MARCH_NT);
  cfg.dynamicSmemBytes = sizeof(MarchSmem<ST, SD>);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // consecutive steps overlap their launches
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_march<MODE, ST, SD, FF, XW>, P, g, mo);
}

template <int MODE, int ST, bool SD, bool FF>
static cudaError_t launch_rows_xw(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  return g.bc_x == BC_WALL ? launch_march<MODE, ST, SD, FF, true>(P, g, mo, st)
                           : launch_march<MODE, ST, SD, FF, false>(P, g, mo, st);
}

template <int MODE, int ST>
static cudaError_t launch_rows_st(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  // the forced order-parameter form changes only the step's f collision (FP32 storage only)
  if constexpr (MODE == MODE_STEP && ST == ST_FP32) {
    if (P.f_forced)
      return P.s_direct ? launch_rows_xw<MODE, ST, true, true>(P, g, mo, st) : launch_rows_xw<MODE, ST, false, true>(P, g, mo, st);
  }
  return P.s_direct ? launch_rows_xw<MODE, ST, true, false>(P, g, mo, st) : launch_rows_xw<MODE, ST, false, false>(P, g, mo, st);
}

}  // namespace lbm
