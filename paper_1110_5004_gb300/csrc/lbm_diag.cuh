// FP64 diagnostics of a set of fields, in one launch.  A block takes up to 8 rows; fixed per-thread strides and fixed
// trees give 12 partials per block, and the block that finishes last folds them in a fixed order.  Results are
// bitwise reproducible.
//
// FP64 runs at about two lanes per cycle and SM here, so the pass is bound by its FP64 instructions (262144
// cells: 75 us with a division and a square root per cell, and eleven block-wide trees per row).  What need not
// be FP64 is not: the clamp, the phase tests and the cell counts are exact in FP32 and integers, FP32 widens by
// integer instructions, the liquid fraction is one fma where 2 phi* is a power of two (dividing by it is then exact),
// |u|^2 is only formed where FP32 rounded up exceeds the largest so far, the root is taken once, and only the
// liquid sum of a row has a tree per row (its largest is the widest chord).
#pragma once
#include <math.h>

#include "lbm_internal.h"

namespace lbm {

constexpr int DIAG_T = 256;
constexpr int DIAG_ROWS = 8;              // most rows of a block
// Rows of a block: about four blocks for each of 152 SMs (a constant, so that the order does not depend on the device).
__host__ __device__ constexpr int diag_rows(int ny) {
  const int r = (ny + 4 * 152 - 1) / (4 * 152);
  return r < DIAG_ROWS ? r : DIAG_ROWS;
}

struct DiagIn {
  const float *phi, *ux, *uy, *p;   // rows of `pitch` elements
  int nx, ny, pitch;
  double phs;                       // phi*
  float phs_f;                      // phi* in FP32, used where `exact`
  float liq;                        // the largest float not above 0.9 phi*
  double half;                      // 1 / (2 phi*)
  int exact;                        // phi* is an FP32 number and 2 phi* a power of two
  int rows;                         // rows of a block
  double* part;                     // 12 partials per block
  double* out;                      // lbm_diag record
  unsigned int* done;               // blocks finished; zero before and after a launch
  long long step;
};

inline DiagIn diag_in(const float* phi, const float* ux, const float* uy, const float* p, int nx, int ny, int pitch, double phs,
                      double* part, double* out, unsigned int* done, long long step) {
  DiagIn d{};
  d.phi = phi;
  d.ux = ux;
  d.uy = uy;
  d.p = p;
  d.nx = nx;
  d.ny = ny;
  d.pitch = pitch;
  d.phs = phs;
  d.phs_f = (float)phs;
  const double t = 0.9 * phs;
  d.liq = (float)t;
  if ((double)d.liq > t) d.liq = nextafterf(d.liq, -INFINITY);
  d.half = 1.0 / (2.0 * phs);
  int e = 0;
  d.exact = (double)d.phs_f == phs && frexp(2.0 * phs, &e) == 0.5 && e > -100 && e < 100;
  d.rows = diag_rows(ny);
  d.part = part;
  d.out = out;
  d.done = done;
  d.step = step;
  return d;
}

// FP32 to FP64 by integer instructions (the conversion runs at the FP64 rate); denormals, infinities and NaN take the
// conversion.
__device__ __forceinline__ double widen64(float v) {
  const unsigned int b = __float_as_uint(v), m = b & 0x7fffffffu;
  if (m - 1u < 0x007fffffu || m >= 0x7f800000u) return (double)v;
  return __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(b << 29));
}

__device__ __forceinline__ double diag_max(double a, double b) { return (a >= b || a != a) ? a : b; }   // NaN propagates

// Tree of one quantity over the block's 256 values v[t] (shared memory), by one warp; the result in lane 0.  The
// order is that of halving the block: t + 128, t + 64, t + 32, then within the warp.
template <bool MAX>
__device__ __forceinline__ double diag_tree(const double* v, int lane) {
  auto op = [](double a, double b) { return MAX ? diag_max(a, b) : a + b; };
  double w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) w[k] = v[k * 32 + lane];
  double s = op(op(op(w[0], w[4]), op(w[2], w[6])), op(op(w[1], w[5]), op(w[3], w[7])));
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) s = op(s, __shfl_down_sync(0xffffffffu, s, k));
  return s;
}

struct DiagSmem {
  double sh[7][DIAG_T];                     // phi, c x, c u_x, c u_y, |u|^2, p in the liquid, p in the gas
  double row_c[DIAG_ROWS][DIAG_T];
  double chord[DIAG_ROWS], total[DIAG_PARTIALS];
  double quot[6];
  int count[2][DIAG_T / 32];
  bool last;
};

static __global__ void __launch_bounds__(DIAG_T) k_diag(const __grid_constant__ DiagIn d) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  DiagSmem& sm = *reinterpret_cast<DiagSmem*>(smem_raw);
  auto& sh = sm.sh;
  auto& row_c = sm.row_c;
  auto& chord = sm.chord;
  auto& total = sm.total;
  auto& quot = sm.quot;
  auto& count = sm.count;
  bool& last = sm.last;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int y0 = blockIdx.x * d.rows, rows = min(d.rows, d.ny - y0);
  // launched as a programmatic dependent of the moment pass
  asm volatile("griddepcontrol.wait;" ::: "memory");
  {
    double phi = 0.0, cx = 0.0, cu = 0.0, cv = 0.0, u2 = 0.0, pl = 0.0, pg = 0.0;
    float u2_low = 0.0f;                    // u2 rounded down
    int nl = 0, ng = 0;
    for (int r = 0; r < rows; ++r) {
      const long long o = (long long)(y0 + r) * d.pitch;
      double c1 = 0.0, xd = t;
      for (int x = t; x < d.nx; x += DIAG_T, xd += DIAG_T) {
        const float phf = d.phi[o + x], uf = d.ux[o + x], vf = d.uy[o + x], pf = d.p[o + x];
        const double ph = widen64(phf), u = widen64(uf), v = widen64(vf), p = widen64(pf);
        double c;
        if (d.exact) {
          c = phf < -d.phs_f ? 0.0 : (phf > d.phs_f ? 1.0 : fma(ph, d.half, 0.5));
        } else {
          c = (ph + d.phs) / (2.0 * d.phs);
          c = c < 0.0 ? 0.0 : (c > 1.0 ? 1.0 : c);
        }
        phi += ph;
        c1 += c;
        cx = fma(c, xd, cx);
        cu = fma(c, u, cu);
        cv = fma(c, v, cv);
        if (!(__fmaf_ru(uf, uf, __fmul_ru(vf, vf)) <= u2_low)) {
          const double q = fma(u, u, v * v);
          u2 = diag_max(u2, q);
          u2_low = __double2float_rd(u2);   // NaN from here on, once there is one
        }
        if (phf > d.liq) {
          pl += p;
          ++nl;
        }
        if (phf < -d.liq) {
          pg += p;
          ++ng;
        }
      }
      row_c[r][t] = c1;
    }
    sh[0][t] = phi;
    sh[1][t] = cx;
    sh[2][t] = cu;
    sh[3][t] = cv;
    sh[4][t] = u2;
    sh[5][t] = pl;
    sh[6][t] = pg;
    nl = __reduce_add_sync(0xffffffffu, nl);
    ng = __reduce_add_sync(0xffffffffu, ng);
    if (lane == 0) {
      count[0][warp] = nl;
      count[1][warp] = ng;
    }
  }
  __syncthreads();
  for (int k = warp; k < 7 + rows; k += DIAG_T / 32) {
    const double* v = k < 7 ? sh[k] : row_c[k - 7];
    const double s = k == 4 ? diag_tree<true>(v, lane) : diag_tree<false>(v, lane);
    if (lane == 0) {
      if (k < 7) total[k] = s;
      else chord[k - 7] = s;
    }
  }
  __syncthreads();
  if (t == 0) {
    double* const q = d.part + (long long)blockIdx.x * DIAG_PARTIALS;
    double c = 0.0, cy = 0.0, wide = 0.0;
    long long nl = 0, ng = 0;
    for (int r = 0; r < rows; ++r) {
      c += chord[r];
      cy = fma(chord[r], (double)(y0 + r), cy);
      wide = diag_max(wide, chord[r]);
    }
    for (int k = 0; k < DIAG_T / 32; ++k) {
      nl += count[0][k];
      ng += count[1][k];
    }
    q[0] = total[0];
    q[1] = c;
    q[2] = total[1];
    q[3] = cy;
    q[4] = total[2];
    q[5] = total[3];
    q[6] = total[4];
    q[7] = total[5];
    q[8] = (double)nl;
    q[9] = total[6];
    q[10] = (double)ng;
    q[11] = wide;                           // widest liquid chord
    __threadfence();
    last = atomicAdd(d.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the partials of all blocks: quantity k by warps k, k + 8; lane l takes blocks l, l + 32, ...
  for (int k = warp; k < DIAG_PARTIALS; k += DIAG_T / 32) {
    const bool max = k == 6 || k == 11;
    double s = 0.0;
    for (unsigned int b = lane; b < gridDim.x; b += 32) {
      const double v = __ldcg(d.part + (long long)b * DIAG_PARTIALS + k);
      s = max ? diag_max(s, v) : s + v;
    }
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
      const double v = __shfl_down_sync(0xffffffffu, s, h);
      s = max ? diag_max(s, v) : s + v;
    }
    if (lane == 0) total[k] = k == 6 ? sqrt(s) : s;
  }
  __syncthreads();
  // the six quotients by six threads: FP64 divisions are long
  if (t < 6) {
    const int num = t < 4 ? 2 + t : (t == 4 ? 7 : 9), den = t < 4 ? 1 : (t == 4 ? 8 : 10);
    quot[t] = total[den] > 0 ? total[num] / total[den] : 0.0;
  }
  __syncwarp();
  if (t == 0) {
    lbm_diag o;
    o.step = d.step;
    o.sum_phi = total[0];
    o.liquid_area = total[1];
    o.centroid_x = quot[0];
    o.centroid_y = quot[1];
    o.vel_x = quot[2];
    o.vel_y = quot[3];
    o.spread_radius = 0.5 * total[11];
    o.max_u = total[6];
    o.p_liquid = quot[4];
    o.p_gas = quot[5];
    o.finite = isfinite(o.sum_phi) && isfinite(o.max_u);
    o.pad = 0;
    *reinterpret_cast<lbm_diag*>(d.out) = o;
    *d.done = 0u;
  }
}

// Launched behind a moment pass on the same stream, which it waits for.  Its blocks are placed while that pass still
// runs, wherever an SM has room: each asks for so much shared memory that no SM takes more than its share.  (They
// piled up on the first SMs that had room, FP64-bound; us a call with the moment pass: 4096 x 152 108 -> 55, 16384 x 64
// 169 -> 111, 74176 x 8 865 -> 322, 1000 x 701 85 -> 74.)
static cudaError_t launch_diag_rows(const DiagIn& d, int sms, cudaStream_t st) {
  static const cudaError_t attr_set =   // once, thread-safely (one GPU per process)
      cudaFuncSetAttribute(k_diag, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_for_cap((int)sizeof(DiagSmem), 1));
  if (attr_set != cudaSuccess) return attr_set;
  const int blocks = (d.ny + d.rows - 1) / d.rows;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(DIAG_T);
  cfg.dynamicSmemBytes = smem_for_cap((int)sizeof(DiagSmem), (blocks + sms - 1) / sms);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_diag, d);
}

}  // namespace lbm
