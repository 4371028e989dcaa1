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
template <int ST, bool SD, int NT>
struct BatchSmem {
  MarchSmem<ST, SD, NT> m;
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
template <int ST, bool SD, bool XW, int NT>
__global__ void __launch_bounds__(NT, march_ctas(NT)) k_batch(const SimDesc* __restrict__ sims, const int4* __restrict__ work,
                                                                int n_work, int parity, unsigned int* __restrict__ next) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  BatchSmem<ST, SD, NT>& sm = *reinterpret_cast<BatchSmem<ST, SD, NT>*>(smem_raw);
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
    for (int k = threadIdx.x; k < (int)(sizeof(Phys2) / 4); k += NT) to[k] = from[k];
    Grid g = d.g;
    const bool odd = ((d.cur0 + parity) & 1) != 0;
    g.src = odd ? d.buf1 : d.buf0;
    g.dst = odd ? const_cast<void*>(d.buf0) : d.buf1;
    if (threadIdx.x == 0) sm.next = (int)(gridDim.x + taken);
    __syncthreads();
    w = __shfl_sync(0xffffffffu, sm.next, 0);   // (uniform to the compiler, which keeps addresses in uniform registers)
    if (sm.m.quit != 0u) {  // a wait ran out in an earlier tile (of any thread: behind its last barrier): not done
      if (threadIdx.x == 0) d.g.give_up.raise();
      __syncthreads();      // sm.next is read above and written for the next tile
      continue;
    }
    march<MODE_STEP, ST, SD, false, XW, false, NT>(sm.P, g, &d.g.give_up, MomentOut{}, it.y, it.z, sm.m, fat, gat);
  }
}

// The tiles work[0, n) of one storage and one form of the mass defect; nt: threads per CTA.
struct BatchPart {
  const SimDesc* sims;
  const int4* work;
  int n, grid, parity, nt;
  unsigned int* next;
  bool sd, xw;
};

template <int ST, bool SD, bool XW, int NT>
static cudaError_t launch_batch_t(const BatchPart& p, cudaStream_t st) {
  static_assert((sizeof(BatchSmem<ST, SD, NT>) + 1024) * march_ctas(NT) <= 233472, "the CTAs of an SM fit its shared memory");
  // set once, thread-safely (one GPU per process)
  static const cudaError_t attr_set =
      cudaFuncSetAttribute(k_batch<ST, SD, XW, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BatchSmem<ST, SD, NT>));
  if (attr_set != cudaSuccess) return attr_set;
  k_batch<ST, SD, XW, NT><<<p.grid, NT, sizeof(BatchSmem<ST, SD, NT>), st>>>(p.sims, p.work, p.n, p.parity, p.next);
  return cudaGetLastError();
}

template <int ST, int NT>
static cudaError_t launch_batch_nt(const BatchPart& p, cudaStream_t st) {
  if (p.sd) return launch_batch_t<ST, true, true, NT>(p, st);
  return p.xw ? launch_batch_t<ST, false, true, NT>(p, st) : launch_batch_t<ST, false, false, NT>(p, st);
}

template <int ST>
static cudaError_t launch_batch_st(const BatchPart& p, cudaStream_t st) {
  if (p.nt == MARCH_NT) return launch_batch_nt<ST, MARCH_NT>(p, st);
  return p.nt == 64 ? launch_batch_nt<ST, 64>(p, st) : launch_batch_nt<ST, 32>(p, st);
}

// (in the storages' translation units)
cudaError_t launch_batch_fp32(const BatchPart& p, cudaStream_t st);
cudaError_t launch_batch_fp16(const BatchPart& p, cudaStream_t st);
cudaError_t launch_batch_bf16(const BatchPart& p, cudaStream_t st);

}  // namespace lbm
