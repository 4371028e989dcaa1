// Device side of the two-distribution D2Q9 multiphase lattice Boltzmann step for sm_103a: state
// layout, population access and the per-cell arithmetic every kernel shares.
//
// State layout in HBM (one simulation, one buffer of a ping-pong pair):
//   19 populations per cell (FP32 storage): f_0..f_8, gbar_0..gbar_8 and f_0lo, post-collision.  They are
//   stored where the next step reads them: population a of the row it streams to,
//     f*_a(x, y) lies in row y + e_a,y at column x, and
//     the reversed population of a link that leaves through a wall in row y at column x + e_a,x (wrapped),
//   so that the populations that stream into cell (x, y) are, for every cell and with any boundaries,
//   population a at row y, column x - e_a,x (wrapped).  The pull needs one row and no wall handling.
//   A row holds blocks of 32 cells (pitch = nx rounded up to 32 columns), in three regions:
//     F  f_0..f_8      G  gbar_0..gbar_8      L  f_0lo (FP32 storage only)
//   population after population inside a block (128 bytes each; 16-bit storage: f_0 in FP32, 128 bytes, then 64
//   bytes each).  So the cells x0 .. x1 of one row are one contiguous piece per region, which the row
//   march copies into shared memory with one bulk copy, and a warp's access to 32 consecutive cells of a
//   population touches at most two blocks (in shared memory: no bank conflict).
//   The rest population f_0 ~ phi is the only O(1) population; it is kept as an unevaluated
//   float pair f_0 + f_0lo so that phi, and through it mu and the surface-tension force, carry
//   ~2^-48 relative precision with FP32 arithmetic.  All other populations are O(mu, u) and need
//   no such care.
//   With the direct mass defect (s_form 1) each buffer also holds, after the populations, two
//   FP32 planes [rho, div(rho u)] of the step that wrote it, each ny rows of `pitch` elements.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace lbm {

constexpr int Q = 9;
constexpr int BC_PERIODIC = 0;
constexpr int BC_WALL = 1;

// D2Q9 ordering: rest, E, N, W, S, NE, NW, SW, SE.
__host__ __device__ constexpr int cx(int a) {
  return a == 1 || a == 5 || a == 8 ? 1 : (a == 3 || a == 6 || a == 7 ? -1 : 0);
}
__host__ __device__ constexpr int cy(int a) {
  return a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0);
}
__host__ __device__ constexpr int opp(int a) {
  return a == 0 ? 0 : (a <= 4 ? ((a + 1) & 3) + 1 : ((a - 3) & 3) + 5);
}
__host__ __device__ constexpr float wgt(int a) {
  return a == 0 ? 4.0f / 9.0f : (a <= 4 ? 1.0f / 9.0f : 1.0f / 36.0f);
}
static_assert(opp(1) == 3 && opp(2) == 4 && opp(3) == 1 && opp(4) == 2, "axis opposites");
static_assert(opp(5) == 7 && opp(6) == 8 && opp(7) == 5 && opp(8) == 6, "diagonal opposites");

// ---- Two cells at a time.  V2 is a pair of FP32 values in a 64-bit register pair, one per cell;
// sm_103a adds, multiplies and fuses both with one instruction, each lane rounded as the scalar
// instruction rounds it.  The stage functions below are written over the value type: float (the
// small-grid tile kernel) or V2 (the row march), with the same operations in the same order, so a
// cell's result does not depend on the kernel that computes it.
struct __align__(8) V2 {
  unsigned long long v;
};
__host__ __device__ __forceinline__ V2 pack2(float a, float b) {
  V2 r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
#else
  union { float f[2]; unsigned long long v; } u = {{a, b}};
  r.v = u.v;
#endif
  return r;
}
__device__ __forceinline__ void unpack2(V2 p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}

// Every floating-point operation of the step is an explicit round-to-nearest instruction, and a product that an addition
// takes is a scalar one (fmul_add), so that no multiply-add is contracted: a cell's arithmetic is the same in every
// kernel, alone or in a batch.
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ V2 fadd(V2 a, V2 b) {
  V2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2 fsub(V2 a, V2 b) {
  V2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// (not where an addition takes the product: fmul_add)
__device__ __forceinline__ V2 fmul(V2 a, V2 b) {
  V2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2 fmad(V2 a, V2 b, V2 c) {
  V2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// A product that an addition follows.  A packed multiply and a packed add in a row were contracted
// into one fma (one-ulp differences from the scalar pair); scalar products keep them apart.
__device__ __forceinline__ float fmul_add(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ V2 fmul_add(V2 a, V2 b) {
  float a0, a1, b0, b1;
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  return pack2(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}
__device__ __forceinline__ float sat_mad(float a, float b, float c) { return __saturatef(fmad(a, b, c)); }
__device__ __forceinline__ V2 sat_mad(V2 a, V2 b, V2 c) {
  float a0, a1, b0, b1, c0, c1;
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  unpack2(c, c0, c1);
  return pack2(sat_mad(a0, b0, c0), sat_mad(a1, b1, c1));
}
// Approximate reciprocal of a normal number (densities and relaxation times), one instruction.
__device__ __forceinline__ float rcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ V2 rcp(V2 a) {
  float x, y;
  unpack2(a, x, y);
  return pack2(rcp(x), rcp(y));
}
template <class V>
__device__ __forceinline__ V zero();
template <>
__device__ __forceinline__ float zero<float>() { return 0.0f; }
template <>
__device__ __forceinline__ V2 zero<V2>() { return V2{0ull}; }

// Scheme constants in FP32, derived once on the host from lbm_params, and the literals the stage
// functions use.  PhysT<float>: literals are immediates.  PhysT<V2>: every constant doubled, so
// that a packed instruction takes it straight from the constant bank.
#define LBM_PHYS_FIELDS(X)                                                                                     \
  X(four_beta)     /* 4 beta */                                                                                \
  X(phi_star) X(inv_2phistar) /* phi*, 1 / (2 phi*) */                                                         \
  X(rho_B) X(drho) /* rho_B, rho_A - rho_B */                                                                  \
  X(ngravity)      /* -g */                                                                                    \
  X(omega_f)       /* 1 / tau_f */                                                                             \
  X(nkappa6)       /* -kappa / 6 (the isotropic Laplacian carries 1/6) */                                      \
  X(rho_prime12)   /* rho' / 12, rho' = drho / (2 phi*) (the isotropic gradient carries 1/12) */               \
  X(s_coef6)       /* rho' theta_M / 6 */                                                                      \
  X(mu3_B) X(mu3_d) /* 3 mu_B, 3 (mu_A - mu_B), mu_X = rho_X cs2 (tau_g_X - 1/2) */                            \
  X(keep_f)        /* 1 - omega_f */                                                                           \
  X(of3gf)         /* omega_f 3 Gamma_f */                                                                     \
  X(hf12)          /* (1 - omega_f / 2) / 12: weight of the forced form's grad(phi) forcing (12 grad phi) */   \
  X(thM6)          /* theta_M / 6: its mobility source from 6 lap(mu) */
#define LBM_LITERALS(X)                                                                                        \
  X(k4, 4.0f) X(km20, -20.0f) X(k3, 3.0f) X(km3, -3.0f) X(k45, 4.5f) X(km15, -1.5f) X(k05, 0.5f)               \
  X(km05, -0.5f) X(k1, 1.0f) X(k6th, 1.0f / 6.0f) X(k12th, 1.0f / 12.0f) X(km12th, -1.0f / 12.0f)              \
  X(k3rd, 1.0f / 3.0f) X(km3rd, -1.0f / 3.0f) X(w0, 4.0f / 9.0f) X(w1, 1.0f / 9.0f) X(w2, 1.0f / 36.0f)        \
  X(nw0, -4.0f / 9.0f) X(nw1, -1.0f / 9.0f) X(nw2, -1.0f / 36.0f) X(kscale, 4096.0f) X(kiscale, 1.0f / 4096.0f)

// Uniform switches of the scheme.
struct PhysFlags {
  int remove_Fa;
  int ch_conv;          // 1: the f collision adds w_a phi div(u) (convective Cahn-Hilliard form)
  int fs_mu;            // 1: F_s = mu grad(phi); 0: F_s = -phi grad(mu)
  int s_direct;         // 1: s = (rho - rho_prev) + div(rho u)_prev from the state's extra planes
  int f_forced;         // 1: forced order-parameter LBE (equilibrium phi Gamma_a)
};
template <class V>
struct PhysT;
template <>
struct PhysT<float> : PhysFlags {
#define X(n) float n;
  LBM_PHYS_FIELDS(X)
#undef X
#define X(n, c) static constexpr float n = c;
  LBM_LITERALS(X)
#undef X
  float kappa, phi_star2, three_gamma_f;   // initial state only
};
template <>
struct PhysT<V2> : PhysFlags {
#define X(n) V2 n;
  LBM_PHYS_FIELDS(X)
#undef X
#define X(n, c) V2 n;
  LBM_LITERALS(X)
#undef X
};
using Phys = PhysT<float>;
using Phys2 = PhysT<V2>;
inline Phys2 widen(const Phys& p) {
  Phys2 r{};
  static_cast<PhysFlags&>(r) = p;
#define X(n) r.n = pack2(p.n, p.n);
  LBM_PHYS_FIELDS(X)
#undef X
#define X(n, c) r.n = pack2(c, c);
  LBM_LITERALS(X)
#undef X
  return r;
}

// ---- Population storage.  FP32: f_0 as the pair f_0 + f_0lo.  FP16 / BF16: the rest population
// f_0 ~ phi stays one float (16-bit rounding of an O(1) value would drift phi by ~1e-4 per step);
// the 17 other populations, all O(mu, u), are 16-bit, stored as value x scale: 2^12 for FP16
// (which maps 1.5e-8 .. 16 onto its normal range), 1 for BF16.
constexpr int ST_FP32 = 0, ST_FP16 = 1, ST_BF16 = 2;
constexpr int A_F0LO = 18;     // population index of f_0lo (FP32 storage)
constexpr int BLK = 32;        // cells per block

__host__ __device__ constexpr long long state_bytes_per_cell(int st) { return st == ST_FP32 ? 4 * 19 : 4 + 2 * 17; }
__host__ __device__ constexpr int elem_bytes(int st) { return st == ST_FP32 ? 4 : 2; }

enum { R_F = 0, R_G = 1, R_L = 2 };   // regions of a row, in this order
__host__ __device__ constexpr int region_of(int a) { return a == A_F0LO ? R_L : (a < Q ? R_F : R_G); }
// Bytes per element of population a, bytes of a region's block, and of the regions before it per block.
__host__ __device__ constexpr int pop_bytes(int st, int a) { return st == ST_FP32 || a == 0 ? 4 : 2; }
__host__ __device__ constexpr int region_block(int st, int r) {
  return r == R_L ? (st == ST_FP32 ? BLK * 4 : 0) : (r == R_F && st != ST_FP32 ? BLK * (4 + 8 * 2) : BLK * 9 * elem_bytes(st));
}
__host__ __device__ constexpr int region_start(int st, int r) {
  return r == R_F ? 0 : (r == R_G ? region_block(st, R_F) : region_block(st, R_F) + region_block(st, R_G));
}
static_assert(region_start(ST_FP32, R_L) + region_block(ST_FP32, R_L) == 76 * BLK && region_start(ST_FP16, R_L) == 38 * BLK, "");
// Byte offset of population a inside its block (lane 0).
__host__ __device__ constexpr int pop_off(int st, int a) {
  return a == A_F0LO ? 0
         : a >= Q ? (a - Q) * BLK * elem_bytes(st)
                  : (st == ST_FP32 ? a * BLK * 4 : (a == 0 ? 0 : BLK * 4 + (a - 1) * BLK * 2));
}

// The waits of the row march for its copies.  They end with the copies; the limit keeps a fault elsewhere from turning
// into a hang.  A launch whose wait runs out raises both words.
struct GiveUp {
  unsigned int* word;   // on the device, kept until the next state (k_init_pop, lbm_restore) or until it is read
  unsigned int* host;   // the same in page-locked memory, which the host reads without a copy; or null
  __device__ __forceinline__ void raise() const {
    *static_cast<volatile unsigned int*>(word) = 1u;
    if (host) *static_cast<volatile unsigned int*>(host) = 1u;
  }
};

struct Grid {
  const void* src;      // post-collision state at t-1 (read)
  void* dst;            // post-collision state at t (write)
  int plane;            // elements per plane of the s_form planes (ny * pitch)
  int row_bytes;        // bytes per population row (the region fits in 2^31 bytes)
  int nblk;             // blocks per region of a row: pitch / 32
  int storage;          // ST_FP32 / ST_FP16 / ST_BF16
  int nx, ny, pitch;
  int bc_x, bc_y;
  int march_nt;         // threads of a row-march CTA
  int tile_w;           // columns per lane of a row-march CTA (a CTA covers two lanes)
  int seg_h;            // rows per segment
  int n_strips;         // CTAs across the grid
  int wait_tries;       // limit of a wait of the row march
  int wait_hold;        // test hook: this tile's rows are never copied (-1: none)
  long long spoff;      // s_form 1: byte offset of the [rho, div(rho u)] planes in src/dst (else 0)
  GiveUp give_up;
};

// Outputs of the moment pass (row-major); each may be null.  fax, fay: the
// additional interfacial force F_a = -u s of Eq. 12 (s by the simulation's s_form), evaluated
// whichever scheme runs.
struct MomentOut {
  float *phi, *rho, *ux, *uy, *p;
  float *fax, *fay;
  int pitch;            // elements per row of every output
};

// Initial fields phi0, ux0, uy0, p0: rows of `pitch` elements; null for zero.
struct InitIn {
  const float* f[4];
  int pitch[4];
};

__host__ __device__ __forceinline__ int wrap(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// Wrap an index that lies within one period of [0, n) (the general case takes a modulo).
__host__ __device__ __forceinline__ int wrap1(int i, int n) {
  if (i < -n || i >= 2 * n) return wrap(i, n);
  return i < 0 ? i + n : (i >= n ? i - n : i);
}

// Byte offsets of column x inside the regions of a row (region starts excluded): for the populations
// of 4 and of 2 bytes (16-bit storage) in F, for G, and for L.
struct ColB {
  int f4, f2, g, l;
};
template <int ST>
__host__ __device__ __forceinline__ ColB col_bytes(int blk, int lane) {
  const int f = blk * region_block(ST, R_F);
  return ColB{f + lane * 4, f + lane * 2, blk * region_block(ST, R_G) + lane * elem_bytes(ST), blk * region_block(ST, R_L) + lane * 4};
}
template <int ST>
__host__ __device__ __forceinline__ ColB col_bytes(int x) {
  return col_bytes<ST>(x >> 5, x & (BLK - 1));
}
// Byte offset of population a at column c from the start of its region.
template <int ST>
__host__ __device__ __forceinline__ int pop_in_region(int a, const ColB& c) {
  return (a == A_F0LO ? c.l : (a >= Q ? c.g : (ST == ST_FP32 || a == 0 ? c.f4 : c.f2))) + pop_off(ST, a);
}
// Byte offset of population a at row offset `row` (row * row_bytes), column c.
template <int ST>
__host__ __device__ __forceinline__ int pop_at(int a, int row, const ColB& c, const Grid& g) {
  return row + region_start(ST, region_of(a)) * g.nblk + pop_in_region<ST>(a, c);
}

// The place of cell (x, y) that keys BF16 stochastic rounding: its byte offset in the row-major
// order of 32-cell blocks that checkpoints use, so the rounding of a value does not depend on
// the order in memory.  pop_key adds the population.
template <int ST>
__host__ __device__ __forceinline__ unsigned int hash_key(int x, int y, const Grid& g) {
  constexpr int B32 = 32 * (int)state_bytes_per_cell(ST);
  return static_cast<unsigned int>(y * (g.pitch / 32 * B32) + (x >> 5) * B32 + (x & 31) * 2);
}
__host__ __device__ constexpr unsigned int pop_key(int a) { return a == 0 ? 0u : 128u + (a - 1) * 64u; }

// Columns x-1, x, x+1 (wrapped).
struct Col3 {
  ColB cm, c0, cq;
};
template <int ST>
__device__ __forceinline__ Col3 col3(int xp, int nx) {
  return Col3{col_bytes<ST>(xp == 0 ? nx - 1 : xp - 1), col_bytes<ST>(xp), col_bytes<ST>(xp == nx - 1 ? 0 : xp + 1)};
}

// Error-free sum of two values: s + e == a + b exactly (round-to-nearest, no contraction).
template <class V>
__device__ __forceinline__ void two_sum(V a, V b, V& s, V& e) {
  s = fadd(a, b);
  const V bb = fsub(s, a);
  e = fadd(fsub(a, fsub(s, bb)), fsub(b, bb));
}

// Population at an address, as stored bits (a float, or a 16-bit value in the low half), and
// their decoding.  A prefetch keeps the bits and decodes them where they are used.  COH: a kernel
// that reads state other CTAs write during the same launch loads through L2 only (ld.global.cg,
// ordered by the memory model); every other kernel takes the read-only path.
template <int ST, bool COH = false>
__device__ __forceinline__ unsigned int ld_raw(const void* __restrict__ base, int a, int off) {
  const char* p = static_cast<const char*>(base) + off;
  if (pop_bytes(ST, a) == 4) {
    const float* q = reinterpret_cast<const float*>(p);
    return __float_as_uint(COH ? __ldcg(q) : __ldg(q));
  }
  const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
  return COH ? __ldcg(q) : __ldg(q);
}

// Decoded populations stay in their storage scale: a 16-bit population holds the value times a
// power of two, and the step carries that scale through its linear arithmetic instead of
// multiplying every value: the sums of S0 and S2 are unscaled once per cell, the collision's
// per-cell constants are scaled once.  Scaling by a power of two is exact, so every result is
// bitwise the one of unscaled arithmetic.
template <int ST>
__device__ __forceinline__ float dec_pop(unsigned int raw, int a) {
  if (pop_bytes(ST, a) == 4) return __uint_as_float(raw);
  const unsigned short r16 = static_cast<unsigned short>(raw);
  return ST == ST_FP16 ? __half2float(__ushort_as_half(r16)) : __bfloat162float(__ushort_as_bfloat16(r16));
}
template <int ST, class V, class K>
__device__ __forceinline__ V to_scale(const K& P, V v) {
  if constexpr (ST == ST_FP16) return fmul(v, P.kscale);
  else return v;
}
template <int ST, class V, class K>
__device__ __forceinline__ V from_scale(const K& P, V v) {
  if constexpr (ST == ST_FP16) return fmul(v, P.kiscale);
  else return v;
}

// BF16 bits of v by stochastic rounding: a pseudo-random 16-bit offset is added to the 16 bits
// that truncation drops, so v rounds away from zero with probability equal to the dropped
// fraction and the rounding error has zero mean.  Round-to-nearest at BF16's 8-bit significand
// biases the gbar populations, which change little from step to step, the same way every step:
// a falling drop's centroid velocity drifted by 3.6 %.  Unbiased rounding of the gbar populations
// keeps it within 0.05 %; the f populations round to nearest (rounding them stochastically as well
// gained nothing, and rounding only them left the 3.6 %).
// The offset is a hash of the value's own bits and its place, so every kernel rounds a
// given value at a given place alike and runs stay deterministic.  NaN and infinity stay NaN and infinity, so a
// diverged state stays non-finite.
// The conversion adds the high and the low half of its third operand to the 16 bits that it drops of the first and the
// second value: what an integer addition to the value's bits gives, with four instructions fewer per value (4096^2: 391 ->
// 371 us a step; 2048 x 512: 35.5 -> 34.2).
__device__ __forceinline__ unsigned int bf16_hash(float v, unsigned int where) {
  // the high half of a product with an odd constant depends on every bit of the other factor
  return (__float_as_uint(v) ^ where) * 0x9e3779b1u;
}
// The bits of lo and hi (at their places) in the low and the high half.
__device__ __forceinline__ unsigned int bf16_stochastic2(float lo, unsigned int at_lo, float hi, unsigned int at_hi) {
  unsigned int d;
  asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;"
      : "=r"(d)
      : "f"(hi), "f"(lo), "r"(__byte_perm(bf16_hash(lo, at_lo), bf16_hash(hi, at_hi), 0x7632)));
  return d;
}
__device__ __forceinline__ unsigned short bf16_stochastic(float v, unsigned int where) {
  unsigned int d;
  asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v), "f"(0.0f), "r"(bf16_hash(v, where)));
  return static_cast<unsigned short>(d >> 16);
}
// 16-bit encoding of population a (already in storage scale).
template <int ST>
__device__ __forceinline__ unsigned short enc_pop(float v, int a, unsigned int key) {
  if (ST == ST_FP16) return __half_as_ushort(__float2half_rn(v));
  if (a >= Q) return bf16_stochastic(v, key + pop_key(a));   // gbar: see bf16_stochastic
  return __bfloat16_as_ushort(__float2bfloat16_rn(v));       // f: round to nearest meets the bound
}

// Where a cell's new populations go: each to the row it streams to, or back as the reversed population
// where it meets a wall.
// XW, YW: walls possible on x, on y.
template <int ST, bool XW = true, bool YW = true>
struct OutCell {
  char* dst;
  int rm, r0, rq;       // byte offsets of rows y-1, y, y+1 (wrapped)
  Col3 c;
  int nblk;
  bool wl, wr, wb, wt;  // x-1, x+1, y-1, y+1 lie beyond a wall
  unsigned int key;     // the cell's place for BF16 rounding
  // byte offset of the place of population A
  template <int A>
  __device__ __forceinline__ int at() const {
    constexpr int ex = A == A_F0LO ? 0 : cx(A % Q), ey = A == A_F0LO ? 0 : cy(A % Q);
    int off = (ey > 0 ? rq : (ey < 0 ? rm : r0)) + region_start(ST, region_of(A)) * nblk + pop_in_region<ST>(A, c.c0);
    if constexpr (ex != 0 || ey != 0) {
      constexpr int B = opp(A % Q) + (A >= Q ? Q : 0);
      const bool hit = (XW && ((ex > 0 && wr) || (ex < 0 && wl))) || (YW && ((ey > 0 && wt) || (ey < 0 && wb)));
      if (hit) off = r0 + region_start(ST, region_of(A)) * nblk + pop_in_region<ST>(B, ex > 0 ? c.cq : (ex < 0 ? c.cm : c.c0));
    }
    return off;
  }
  template <int A>
  __device__ __forceinline__ void put(float v) const {
    char* p = dst + at<A>();
    if (pop_bytes(ST, A) == 4) *reinterpret_cast<float*>(p) = v;
    else *reinterpret_cast<unsigned short*>(p) = enc_pop<ST>(v, A, key);
  }
};
template <int ST, bool XW = true, bool YW = true>
__device__ __forceinline__ OutCell<ST, XW, YW> out_cell(const Grid& g, int x, int y) {
  OutCell<ST, XW, YW> o;
  o.dst = static_cast<char*>(g.dst);
  o.r0 = y * g.row_bytes;
  o.rm = y == 0 ? (g.ny - 1) * g.row_bytes : o.r0 - g.row_bytes;
  o.rq = y == g.ny - 1 ? 0 : o.r0 + g.row_bytes;
  o.c = col3<ST>(x, g.nx);
  o.nblk = g.nblk;
  o.wl = g.bc_x == BC_WALL && x == 0;
  o.wr = g.bc_x == BC_WALL && x == g.nx - 1;
  o.wb = g.bc_y == BC_WALL && y == 0;
  o.wt = g.bc_y == BC_WALL && y == g.ny - 1;
  o.key = hash_key<ST>(x, y, g);
  return o;
}

// The populations FIRST .. FIRST + 8 (f or gbar) that stream into the cell at columns c of the row at byte offset
// `row`, as stored bits.
template <int ST, int FIRST, bool COH = false>
__device__ __forceinline__ void gather9(const Grid& g, const Col3& c, int row, unsigned int v[Q]) {
#pragma unroll
  for (int a = 0; a < Q; ++a)
    v[a] = ld_raw<ST, COH>(g.src, FIRST + a,
                           pop_at<ST>(FIRST + a, row, cx(a) == 1 ? c.cm : (cx(a) == -1 ? c.cq : c.c0), g));
}

// ---- Per-cell stage arithmetic, shared by every step kernel, so that a cell's result does not
// depend on the kernel that computes it.  Stencil arguments point at the cell's column in rows s
// (south), 0 and n (north); [-1] and [1] are the west and east neighbours.

// Isotropic gradient of a 3x3 stencil, times 12:
//   12 dq/dx = 4 (E - W) + (NE - NW) + (SE - SW) = 4 (E - W) + (d1 - d2)
//   12 dq/dy = 4 (N - S) + (NE - SE) + (NW - SW) = 4 (N - S) + (d1 + d2),  d1 = NE - SW, d2 = NW - SE
template <class V, class K>
__device__ __forceinline__ void grad12(const K& P, const V* s, const V* c, const V* n, V& gx, V& gy) {
  const V d1 = fsub(n[1], s[-1]), d2 = fsub(n[-1], s[1]);
  gx = fmad(P.k4, fsub(c[1], c[-1]), fsub(d1, d2));
  gy = fmad(P.k4, fsub(n[0], s[0]), fadd(d1, d2));
}

// Per-cell record carried from S2 to S3.
template <class V>
struct RecT {
  V phi, mu, ux, uy, Fx, Fy;
  V mrx3, mry3;         // -(grad rho) / 3
  V og;                 // omega_g = 1 / tau_g(phi)
  V ogr3;               // omega_g rho / 3
  V gx12, gy12;         // forced order-parameter form: 12 grad(phi)
  V lmu6;               // and 6 lap(mu)
};

constexpr int NF = Q + 1;    // gathered f_0..f_8 and f_0lo

// S0: phi = sum_a f_a as an unevaluated pair hi + lo (fp[0..8] f_0..f_8, fp[9] f_0lo).
// fp[1..8] in storage scale.
template <int ST, class V, class K>
__device__ __forceinline__ void phi_pair(const K& P, const V fp[NF], V& hi, V& lo) {
  const V s8 = fadd(fadd(fadd(fp[1], fp[2]), fadd(fp[3], fp[4])), fadd(fadd(fp[5], fp[6]), fadd(fp[7], fp[8])));
  const V small = fadd(fp[Q], from_scale<ST>(P, s8));
  two_sum(fp[0], small, hi, lo);
}

// S1: mu = theta'(phi) - kappa lap(phi) (Eq. 1) from the phi pair's 3x3 neighbourhood.
template <class V, class K>
__device__ __forceinline__ V chem_potential(const K& P, const V* hs, const V* h0, const V* hn, const V* ls, const V* l0,
                                            const V* ln) {
  const V H = h0[0], L = l0[0];
  // differences from the centre: exact for neighbouring values of like magnitude; the low
  // words are tiny and are summed directly
  const V dax = fadd(fadd(fsub(h0[1], H), fsub(hn[0], H)), fadd(fsub(h0[-1], H), fsub(hs[0], H)));
  const V ddg = fadd(fadd(fsub(hn[1], H), fsub(hn[-1], H)), fadd(fsub(hs[-1], H), fsub(hs[1], H)));
  const V lax = fadd(fadd(l0[1], ln[0]), fadd(l0[-1], ls[0]));
  const V ldg = fadd(fadd(ln[1], ln[-1]), fadd(ls[-1], ls[1]));
  const V lap6 = fmad(P.km20, L, fmad(P.k4, fadd(dax, lax), fadd(ddg, ldg)));   // 6 lap(phi)
  const V ph = fadd(H, L);
  const V dm = fadd(fsub(H, P.phi_star), L), dp = fadd(fadd(H, P.phi_star), L);
  return fmad(P.nkappa6, lap6, fmul(fmul(fmul(P.four_beta, ph), dm), dp));
}

// 6 lap(q) of the isotropic 9-point Laplacian.
template <class V, class K>
__device__ __forceinline__ V lap6_of(const K& P, const V* s, const V* c, const V* n) {
  return fmad(P.km20, c[0], fmad(P.k4, fadd(fadd(c[1], n[0]), fadd(c[-1], s[0])), fadd(fadd(n[1], n[-1]), fadd(s[-1], s[1]))));
}

// Density of a phi value (clamped linear, Eq. 4).
template <class V, class K>
__device__ __forceinline__ V density(const K& P, V ph) {
  return fmad(sat_mad(ph, P.inv_2phistar, P.k05), P.drho, P.rho_B);
}

// S2: density, surface and body forces, velocity (the second-order scheme of Eq. 8, F_a removed
// or not) and pressure of a cell from phi, 12 grad(phi), 12 grad(mu), mu, the mass defect s (zero
// unless F_a is removed) and the pulled gbar populations (in storage scale).
template <class V>
struct S2Out {
  V rho, cl, fsx, fsy, gy, rrho, ux, uy, rx, ry, p;
};
template <int ST, class V, class K>
__device__ __forceinline__ S2Out<V> s2_cell(const K& P, V ph, V gphx, V gphy, V gmx, V gmy, V mu0, V sdef, const V gb[Q]) {
  S2Out<V> o;
  o.cl = sat_mad(ph, P.inv_2phistar, P.k05);            // clamp((phi + phi*) / (2 phi*))
  o.rho = fmad(o.cl, P.drho, P.rho_B);
  const V q = P.fs_mu ? mu0 : ph, q12 = fmul(q, P.fs_mu ? P.k12th : P.km12th);   // F_s = mu grad phi, or -phi grad mu
  o.fsx = fmul_add(q12, P.fs_mu ? gphx : gmx);
  o.fsy = fmul_add(q12, P.fs_mu ? gphy : gmy);
  o.gy = fmul_add(P.ngravity, o.rho);
  const V s13 = fadd(gb[1], gb[3]), d13 = fsub(gb[1], gb[3]);
  const V s24 = fadd(gb[2], gb[4]), d24 = fsub(gb[2], gb[4]);
  const V s57 = fadd(gb[5], gb[7]), d57 = fsub(gb[5], gb[7]);
  const V s68 = fadd(gb[6], gb[8]), d86 = fsub(gb[8], gb[6]);
  const V m0g = from_scale<ST>(P, fadd(fadd(fadd(gb[0], s13), fadd(s24, s57)), s68));
  const V jx = from_scale<ST>(P, fadd(fadd(d13, d57), d86));
  const V jy = from_scale<ST>(P, fsub(fadd(d24, d57), d86));
  o.rrho = rcp(o.rho);
  const V rden = rcp(fmad(P.km05, sdef, o.rho));        // the density itself where F_a stays (s = 0)
  o.ux = fmul(fmad(P.k3, jx, fmul(P.k05, o.fsx)), rden);
  o.uy = fmul(fmad(P.k3, jy, fmul(P.k05, fadd(o.fsy, o.gy))), rden);
  o.rx = fmul(P.rho_prime12, gphx);                     // grad rho
  o.ry = fmul(P.rho_prime12, gphy);
  o.p = fmad(fmad(o.ux, o.rx, fmul(o.uy, o.ry)), P.k6th, m0g);
  return o;
}

// The record S3 needs from S2 (the forced order-parameter fields are set by the caller).
template <class V, class K>
__device__ __forceinline__ void s2_record(const K& P, const S2Out<V>& o, V ph, V mu0, V sdef, RecT<V>& r) {
  r.phi = ph;
  r.mu = mu0;
  r.ux = o.ux;
  r.uy = o.uy;
  const V fy = fadd(o.fsy, o.gy);
  r.Fx = P.remove_Fa ? fmad(o.ux, sdef, o.fsx) : o.fsx;
  r.Fy = P.remove_Fa ? fmad(o.uy, sdef, fy) : fy;
  r.mrx3 = fmul(P.km3rd, o.rx);
  r.mry3 = fmul(P.km3rd, o.ry);
  const V muv3 = fmad(o.cl, P.mu3_d, P.mu3_B);          // 3 mu(phi)
  r.og = rcp(fmad(muv3, o.rrho, P.k05));                // 1 / tau_g(phi)
  r.ogr3 = fmul(r.og, fmul(o.rho, P.k3rd));
}

// S3: phi div(u) of the convective Cahn-Hilliard source from u_x rows (xs, x0, xn) and u_y rows
// (ys, yn): 12 d(ux)/dx = 4 (E - W) + (NE - SW) - (NW - SE), 12 d(uy)/dy = 4 (N - S) + (NE - SW) + (NW - SE).
template <class V, class K>
__device__ __forceinline__ V phi_div_u(const K& P, V phi, const V* xs, const V* x0, const V* xn, const V* ys, const V* yn) {
  const V dux = fmad(P.k4, fsub(x0[1], x0[-1]), fsub(fsub(xn[1], xs[-1]), fsub(xn[-1], xs[1])));
  const V duy = fmad(P.k4, fsub(yn[0], ys[0]), fadd(fsub(yn[1], ys[-1]), fsub(yn[-1], ys[1])));
  return fmul_add(phi, fmul(fadd(dux, duy), P.k12th));
}

// Both collisions at one cell.  With Gamma_a = omega_a(u) = w_a (1 + poly_a),
// poly_a = 3 e.u + 4.5 (e.u)^2 - 1.5 u.u, gmw_a = Gamma_a - w_a = w_a poly_a, D = F - grad psi:
//   g^eq_a = w_a p + (rho / 3) gmw_a
//   S_a    = (e_a - u).[F Gamma_a - gmw_a grad psi] = w_a (e_a.F - u.F) + gmw_a (e_a.D - u.D)
//   gbar*_a = (1 - omega_g) gbar_a + omega_g g^eq_a + (1 - omega_g / 2) S_a
//   f*_a   = (1 - omega_f) f_a + omega_f w_a (3 Gamma_f mu + phi poly_a) + w_a phi div(u)   (a > 0)
// or, in the forced order-parameter form (FF), with h = 1 - omega_f / 2:
//   f*_a   = (1 - omega_f) f_a + Gamma_a [omega_f phi + h (e_a - u).grad phi + theta_M lap mu]
//            + w_a phi div(u)
// The weight-class products are formed once per cell (class 0: rest, 1: axis, 2: diagonal).  A
// direction and its opposite share e.v up to the sign, which goes into constants and operand order
// (packed instructions have no free negation); each result is exactly that of the plain formula.
template <class V>
struct CollideC {
  V e[4], F[4], D[4];    // u, F, D projected on directions 1, 2, 5, 8
  V m15uu, nuD;
  V wuF[3];              // -w_c u.F
  V A[3];                // omega_g w_c p
  V ogr3, keep_g, src_g;
  V ofwg[3];             // omega_f w_c 3 Gamma_f mu
  V ofwp[3];             // omega_f w_c phi
  V hg[4], c0, ofp;      // FF: h grad(phi) projections; theta_M lap mu - h u.grad phi; omega_f phi
  V wphiD[3];            // FF: w_c phi div(u)
};

// PART: COLLIDE_BOTH, or only the gbar (COLLIDE_G) or only the f (COLLIDE_F) populations, each
// computed exactly as in the joint form (the small-grid kernel gives them to two threads).
constexpr int COLLIDE_BOTH = 0, COLLIDE_F = 1, COLLIDE_G = 2;

// Direction A = +e or -e (NEG) of the projection index I (directions 1, 2, 5, 8).
template <int ST, int A, int I, bool NEG, bool FF, int PART, class V, class K, class Out>
__device__ __forceinline__ void collide_dir(const K& P, const CollideC<V>& k, const V f[Q], const V gb[Q], const Out& out,
                                            V& fsum, V& nofeq) {
  constexpr int C = A <= 4 ? 1 : 2;
  const V w = C == 1 ? P.w1 : P.w2, nw = C == 1 ? P.nw1 : P.nw2;
  const V eu = k.e[I];
  // poly(-e) = 4.5 eu^2 - 3 eu + m15uu, with the rounding of eu -> -eu
  const V poly = NEG ? fmad(eu, fmad(P.k45, eu, P.km3), k.m15uu) : fmad(eu, fmad(P.k45, eu, P.k3), k.m15uu);
  const V gmw = FF ? fmul_add(w, poly) : fmul(w, poly);
  if (PART != COLLIDE_F) {
    const V t1w = fmad(NEG ? nw : w, k.F[I], k.wuF[C]);
    const V t2 = NEG ? fsub(k.nuD, k.D[I]) : fadd(k.D[I], k.nuD);
    const V S = fmad(gmw, t2, t1w);
    out.template put<Q + A>(fmad(k.src_g, S, fmad(k.ogr3, gmw, fmad(k.keep_g, gb[A], k.A[C]))));
  }
  if (PART != COLLIDE_G) {
    V ofeq;
    if constexpr (FF) {
      const V Ga = fadd(w, gmw);                                                // Gamma_a
      const V ta = NEG ? fsub(k.c0, k.hg[I]) : fadd(k.hg[I], k.c0);             // h (e_a - u).grad phi + theta_M lap mu
      ofeq = fmad(Ga, fadd(ta, k.ofp), k.wphiD[C]);
    } else {
      ofeq = fmad(k.ofwp[C], poly, k.ofwg[C]);
    }
    fsum = fadd(fsum, f[A]);
    nofeq = fsub(nofeq, ofeq);
    out.template put<A>(fmad(P.keep_f, f[A], ofeq));
  }
}

// Collision of both distributions at one cell and store of the post-collision populations.
// f[] holds f_1..f_8 (index 0 unused), gb[] gbar_0..gbar_8; gpx12/gpy12 are 12 grad p.
// phiD = phi div(u) (convective form) or 0: the f collision adds w_a phiD to direction a.
template <int ST, bool FF, int PART = COLLIDE_BOTH, class V, class K, class Out>
__device__ __forceinline__ void collide_store(const K& P, const RecT<V>& r, V p, V gpx12, V gpy12, V phi_hi, V phi_lo,
                                              V phiD, const V f[Q], const V gb[Q], const Out& out) {
  CollideC<V> k;
  k.e[0] = r.ux;
  k.e[1] = r.uy;
  k.e[2] = fadd(r.ux, r.uy);
  k.e[3] = fsub(r.ux, r.uy);
  k.m15uu = fmul(P.km15, fmad(r.ux, r.ux, fmul(r.uy, r.uy)));
  if (PART != COLLIDE_F) {
    k.F[0] = r.Fx;
    k.F[1] = r.Fy;
    k.F[2] = fadd(r.Fx, r.Fy);
    k.F[3] = fsub(r.Fx, r.Fy);
    // grad psi = grad p - cs2 grad rho
    k.D[0] = fsub(r.Fx, fmad(gpx12, P.k12th, r.mrx3));
    k.D[1] = fsub(r.Fy, fmad(gpy12, P.k12th, r.mry3));
    k.D[2] = fadd(k.D[0], k.D[1]);
    k.D[3] = fsub(k.D[0], k.D[1]);
    const V uD = fmad(r.ux, k.D[0], fmul(r.uy, k.D[1]));
    k.nuD = fsub(zero<V>(), uD);
    const V uF = fmad(r.ux, r.Fx, fmul(r.uy, r.Fy));
    k.wuF[0] = fmul(P.nw0, uF);
    k.wuF[1] = fmul(P.nw1, uF);
    k.wuF[2] = fmul(P.nw2, uF);
    // terms added to a stored (16-bit: scaled) population carry the storage scale
    const V ogp = fmul(r.og, p);
    k.A[0] = to_scale<ST>(P, fmul(P.w0, ogp));
    k.A[1] = to_scale<ST>(P, fmul(P.w1, ogp));
    k.A[2] = to_scale<ST>(P, fmul(P.w2, ogp));
    k.ogr3 = to_scale<ST>(P, r.ogr3);
    k.keep_g = fsub(P.k1, r.og);
    k.src_g = to_scale<ST>(P, fmad(P.km05, r.og, P.k1));
    // direction 0
    const V gmw = fmul(P.w0, k.m15uu);
    const V S = fmad(gmw, k.nuD, k.wuF[0]);
    out.template put<Q>(fmad(k.src_g, S, fmad(k.ogr3, gmw, fmad(k.keep_g, gb[0], k.A[0]))));
  }
  if (PART != COLLIDE_G) {
    const V ofg = fadd(fmul_add(P.of3gf, r.mu), phiD), ofp = fmul_add(P.omega_f, r.phi);
    k.ofwg[1] = to_scale<ST>(P, fmul(P.w1, ofg));
    k.ofwg[2] = to_scale<ST>(P, fmul(P.w2, ofg));
    k.ofwp[1] = to_scale<ST>(P, fmul(P.w1, ofp));
    k.ofwp[2] = to_scale<ST>(P, fmul(P.w2, ofp));
    if constexpr (FF) {
      const V hx = fmul_add(P.hf12, r.gx12), hy = fmul_add(P.hf12, r.gy12);
      k.hg[0] = hx;
      k.hg[1] = hy;
      k.hg[2] = fadd(hx, hy);
      k.hg[3] = fsub(hx, hy);
      k.c0 = fsub(fmul_add(P.thM6, r.lmu6), fmad(r.ux, hx, fmul(r.uy, hy)));
      k.ofp = ofp;
      k.wphiD[1] = fmul(P.w1, phiD);
      k.wphiD[2] = fmul(P.w2, phiD);
    }
  }
  V fsum = zero<V>(), nofeq = zero<V>();   // sums over a > 0 of f_a and of -(omega_f f^eq_a + w_a phiD)
  collide_dir<ST, 1, 0, false, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 2, 1, false, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 3, 0, true, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 4, 1, true, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 5, 2, false, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 6, 3, true, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 7, 2, true, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  collide_dir<ST, 8, 3, false, FF, PART>(P, k, f, gb, out, fsum, nofeq);
  // f_0 = phi - sum_{a>0} f_a and omega_f (f_0^eq - f_0) = omega_f sum_{a>0} f_a - sum omega_f f^eq_a;
  // the directions a > 0 carry w_a phiD of the source inside nofeq, so the rest gets
  // phiD - (5/9) phiD = w_0 phiD by adding phiD:
  // f*_0 = phi_hi + [(phi_lo - sum f_a) + (omega_f sum f_a - sum (omega_f f^eq_a + w_a phiD)) + phiD].
  // Only small terms are rounded before the one error-free sum with the O(1) high word.
  if (PART == COLLIDE_G) return;
  fsum = from_scale<ST>(P, fsum);          // back from the storage scale (exact)
  nofeq = from_scale<ST>(P, nofeq);
  V hi, lo;
  V small = fadd(fsub(phi_lo, fsum), fmad(P.omega_f, fsum, nofeq));
  // the forced form changes phi by theta_M lap mu (+ phiD) in the collision
  if constexpr (FF) small = fadd(small, fmul_add(P.thM6, r.lmu6));
  two_sum(phi_hi, fadd(small, phiD), hi, lo);
  if (ST == ST_FP32) {
    out.template put<0>(hi);
    out.template put<A_F0LO>(lo);
  } else {
    out.template put<0>(fadd(hi, lo));
  }
}

}  // namespace lbm
