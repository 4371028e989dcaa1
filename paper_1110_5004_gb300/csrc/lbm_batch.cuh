// The batch kernel: the row march over a work list of tiles of many simulations.  Each storage is compiled in a
// translation unit of its own (lbm_batch_fp32.cu, ...).
#pragma once
#include "lbm_internal.h"
#include "lbm_march.cuh"

namespace lbm {

struct SimDesc {
  Phys2 P;
  Grid g;                 // src/dst unused; buffers below
  const void* buf0;
  void* buf1;
  int cur0;               // buffer holding the state when the graph replay starts
  int pad;
};
static_assert(sizeof(Phys2) % 4 == 0, "copied in words");

// The row march's shared memory and the constants of the tile's member, from which its packed
// instructions read them (a kernel parameter cannot differ between CTAs).
template <int ST, bool SD>
struct BatchSmem {
  MarchSmem<ST, SD> m;
  Phys2 P;
  int next;               // the tile after this one
};

// One storage and one form of the mass defect per launch: a kernel that held the march of all three storages
// did not fit 255 registers (1.2-1.9 KB of spills per thread).  XW: some member may have walls on x.
//
// A CTA takes its first tile by its index and further ones from a counter, the list being in order of falling
// height: tiles differ in it, and CTAs that share no SM run faster, so that fixed rounds left CTAs idle (us a
// step, FP32 and BF16: 48 members 184 and 194 -> 179 and 187, 256 members 1036 and 1028 -> 971 and 997; since the march
// has one row body, which left no spills here, 171 and 171, 935 and 947).  next: the counter, zero before and
// after a launch.
template <int ST, bool SD, bool XW>
__global__ void __launch_bounds__(MARCH_NT, MARCH_CTAS) k_batch(const SimDesc* __restrict__ sims, const int4* __restrict__ work,
                                                                int n_work, int parity, unsigned int* __restrict__ next) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  BatchSmem<ST, SD>& sm = *reinterpret_cast<BatchSmem<ST, SD>*>(smem_raw);
  march_init(sm.m);
  StageAt fat, gat;
  for (int w = blockIdx.x; w < n_work;) {
    unsigned int taken = 0;
    if (threadIdx.x == 0) {
      taken = atomicAdd(next, 1u);
      if (taken == n_work - 1u) *next = 0u;   // one addition per tile: this was the last
    }
    const int4 it = work[w];
    const SimDesc& d = sims[it.x];
    const unsigned int* from = reinterpret_cast<const unsigned int*>(&d.P);
    unsigned int* to = reinterpret_cast<unsigned int*>(&sm.P);
    for (int k = threadIdx.x; k < (int)(sizeof(Phys2) / 4); k += MARCH_NT) to[k] = from[k];
    Grid g = d.g;
    const bool odd = ((d.cur0 + parity) & 1) != 0;
    g.src = odd ? d.buf1 : d.buf0;
    g.dst = odd ? const_cast<void*>(d.buf0) : d.buf1;
    if (threadIdx.x == 0) sm.next = (int)(gridDim.x + taken);
    __syncthreads();
    w = __shfl_sync(0xffffffffu, sm.next, 0);   // (uniform to the compiler, which keeps addresses in uniform registers)
    if (sm.m.quit != 0u) {  // a wait ran out in an earlier tile (of any thread: behind its last barrier): not done
      if (threadIdx.x == 0) d.g.wait.raise();
      __syncthreads();      // sm.next is read above and written for the next tile
      continue;
    }
    march<MODE_STEP, ST, SD, false, XW, false>(sm.P, g, &d.g.wait, MomentOut{}, it.y, it.z, sm.m, fat, gat);
  }
}

template <int ST, bool SD, bool XW>
static cudaError_t launch_batch_t(const SimDesc* sims, const int4* work, int n, int grid, int parity, unsigned int* next, cudaStream_t st) {
  // set once, thread-safely (one GPU per process)
  static const cudaError_t attr_set =
      cudaFuncSetAttribute(k_batch<ST, SD, XW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BatchSmem<ST, SD>));
  if (attr_set != cudaSuccess) return attr_set;
  k_batch<ST, SD, XW><<<grid, MARCH_NT, sizeof(BatchSmem<ST, SD>), st>>>(sims, work, n, parity, next);
  return cudaGetLastError();
}

// The tiles work[0, n) of members of one storage and one form of the mass defect.
template <int ST>
static cudaError_t launch_batch_st(const SimDesc* sims, const int4* work, int n, int grid, int parity, unsigned int* next, bool sd,
                                   bool xw, cudaStream_t st) {
  if (sd) return launch_batch_t<ST, true, true>(sims, work, n, grid, parity, next, st);
  return xw ? launch_batch_t<ST, false, true>(sims, work, n, grid, parity, next, st)
            : launch_batch_t<ST, false, false>(sims, work, n, grid, parity, next, st);
}

// (in the storages' translation units)
cudaError_t launch_batch_fp32(const SimDesc*, const int4*, int n, int grid, int parity, unsigned int* next, bool sd, bool xw, cudaStream_t st);
cudaError_t launch_batch_fp16(const SimDesc*, const int4*, int n, int grid, int parity, unsigned int* next, bool sd, bool xw, cudaStream_t st);
cudaError_t launch_batch_bf16(const SimDesc*, const int4*, int n, int grid, int parity, unsigned int* next, bool sd, bool xw, cudaStream_t st);

}  // namespace lbm
