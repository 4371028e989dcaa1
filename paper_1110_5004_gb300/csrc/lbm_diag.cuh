// FP64 diagnostics of a set of fields, in one launch.  One block per row, fixed per-thread stride and fixed
// tree -> 12 partials per row; the block that finishes last folds the rows in a fixed order.  Results are bitwise
// reproducible.
//
// FP64 runs at a small fraction of the FP32 rate here, so the row pass is bound by its FP64 instructions (262144
// cells: 75 us with a division and a square root per cell, and 88 barriers per row in the trees).  What need not
// be FP64 is not: the clamp, the phase tests and the cell counts are exact in FP32 and integers, the liquid
// fraction is one fma where 2 phi* is a power of two (dividing by it is then exact), the square root is taken of a
// row's largest |u|^2, and a tree is three levels across the eight warps' values (by one warp per quantity) and
// five of warp shuffles.
#pragma once
#include <math.h>

#include "lbm_internal.h"

namespace lbm {

constexpr int DIAG_T = 256;

struct DiagIn {
  const float *phi, *ux, *uy, *p;   // rows of `pitch` elements
  int nx, ny, pitch;
  double phs;                       // phi*
  float phs_f;                      // phi* in FP32, used where `exact`
  float liq;                        // the largest float not above 0.9 phi*
  double half;                      // 1 / (2 phi*)
  int exact;                        // phi* is an FP32 number and 2 phi* a power of two
  double* part;                     // ny x 12 partials
  double* out;                      // lbm_diag record
  unsigned int* done;               // rows finished; zero before and after a launch
  const unsigned int* gave_up;      // or null
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
  d.part = part;
  d.out = out;
  d.done = done;
  d.step = step;
  return d;
}

// FP32 to FP64 by integer instructions (the conversion runs at the FP64 rate); zeros, denormals, infinities and NaN
// take the conversion.
__device__ __forceinline__ double widen64(float v) {
  const unsigned int b = __float_as_uint(v), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u) return (double)v;
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
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

static __global__ void __launch_bounds__(DIAG_T) k_diag(const __grid_constant__ DiagIn d) {
  __shared__ double sh[DIAG_PARTIALS][DIAG_T];
  __shared__ bool last;
  const int y = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // launched as a programmatic dependent of the moment pass
  asm volatile("griddepcontrol.wait;" ::: "memory");
  {
    const long long o = (long long)y * d.pitch;
    double phi = 0.0, c1 = 0.0, cx = 0.0, xd = t, cu = 0.0, cv = 0.0, u2 = 0.0, pl = 0.0, pg = 0.0;
    int nl = 0, ng = 0;
    for (int x = t; x < d.nx; x += DIAG_T, xd += DIAG_T) {
      const float phf = d.phi[o + x], pf = d.p[o + x];
      const double ph = widen64(phf), u = widen64(d.ux[o + x]), v = widen64(d.uy[o + x]), p = widen64(pf);
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
      const double q = fma(u, u, v * v);
      if (!(q <= u2)) u2 = q;
      if (phf > d.liq) {
        pl += p;
        ++nl;
      }
      if (phf < -d.liq) {
        pg += p;
        ++ng;
      }
    }
    sh[0][t] = phi;
    sh[1][t] = c1;
    sh[2][t] = cx;
    sh[4][t] = cu;
    sh[5][t] = cv;
    sh[6][t] = u2;
    sh[7][t] = pl;
    sh[8][t] = nl;
    sh[9][t] = pg;
    sh[10][t] = ng;
  }
  __syncthreads();
  double* const r = d.part + (long long)y * DIAG_PARTIALS;
  for (int k = warp; k < 11; k += 8) {
    if (k == 3) continue;
    double s = k == 6 ? diag_tree<true>(sh[k], lane) : diag_tree<false>(sh[k], lane);
    if (k == 6) s = sqrt(s);
    if (lane == 0) r[k] = s;
    if (lane == 0 && k == 1) r[3] = s * (double)y;   // sum(c y) of a row
  }
  if (t == 32) r[11] = 0.0;
  __syncthreads();
  if (t == 0) {
    __threadfence();
    last = atomicAdd(d.done, 1u) == (unsigned int)(d.ny - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double acc[DIAG_PARTIALS] = {0};
  for (int row = t; row < d.ny; row += DIAG_T) {
    const double* q = d.part + (long long)row * DIAG_PARTIALS;
#pragma unroll
    for (int k = 0; k < 11; ++k) {
      const double v = __ldcg(q + k);
      if (k == 6) {
        if (!(v <= acc[6])) acc[6] = v;
      } else {
        acc[k] += v;
      }
      if (k == 1 && !(v <= acc[11])) acc[11] = v;   // widest liquid chord
    }
  }
#pragma unroll
  for (int k = 0; k < DIAG_PARTIALS; ++k) sh[k][t] = acc[k];
  __syncthreads();
  __shared__ double total[DIAG_PARTIALS];
  for (int k = warp; k < DIAG_PARTIALS; k += 8) {
    const double s = (k == 6 || k == 11) ? diag_tree<true>(sh[k], lane) : diag_tree<false>(sh[k], lane);
    if (lane == 0) total[k] = s;
  }
  __syncthreads();
  if (t == 0) {
    lbm_diag o;
    o.step = d.step;
    o.sum_phi = total[0];
    o.liquid_area = total[1];
    const double sc = total[1];
    o.centroid_x = sc > 0 ? total[2] / sc : 0.0;
    o.centroid_y = sc > 0 ? total[3] / sc : 0.0;
    o.vel_x = sc > 0 ? total[4] / sc : 0.0;
    o.vel_y = sc > 0 ? total[5] / sc : 0.0;
    o.spread_radius = 0.5 * total[11];
    o.max_u = total[6];
    o.p_liquid = total[8] > 0 ? total[7] / total[8] : 0.0;
    o.p_gas = total[10] > 0 ? total[9] / total[10] : 0.0;
    o.finite = isfinite(o.sum_phi) && isfinite(o.max_u) && (!d.gave_up || *d.gave_up == 0u);
    o.pad = 0;
    *reinterpret_cast<lbm_diag*>(d.out) = o;
    *d.done = 0u;
  }
}

// dependent: launched behind a moment pass on the same stream, which it waits for.
inline cudaError_t launch_diag_rows(const DiagIn& d, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.ny);
  cfg.blockDim = dim3(DIAG_T);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_diag, d);
}

}  // namespace lbm
