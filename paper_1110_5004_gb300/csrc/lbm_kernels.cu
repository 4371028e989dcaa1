// Kernels of the two-distribution D2Q9 multiphase LBM: fused step, moments, initial state and
// FP64 diagnostics, with their launchers.
#include <math.h>

#include <utility>

#include "lbm_diag.cuh"
#include "lbm_internal.h"

namespace lbm {

// ------------------------------------------------------------------ fused step

cudaError_t launch_step(const Phys2& P, const Grid& g, cudaStream_t st) {
  switch (g.storage) {
    case ST_FP32: return launch_step_fp32(P, g, st);
    case ST_FP16: return launch_step_fp16(P, g, st);
    case ST_BF16: return launch_step_bf16(P, g, st);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------------ initial state
// State that streams into f = f^eq(phi0, mu0, u0), gbar = g^eq(p0, rho0, u0): each cell stores its own 18
// equilibria where it will read them, population a in its row at column x - e_a,x.
template <int ST>
__global__ void k_init_pop(Phys P, Grid g, InitIn in) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  // a new state: the old one's give-up words are cleared, at the end, where the look at one has arrived
  const bool first = x == 0 && blockIdx.y == 0;
  const unsigned int stale = first ? *static_cast<volatile unsigned int*>(g.give_up.word) : 0u;
  if (x >= g.nx) return;
  const Col3 col = col3<ST>(x, g.nx);
  // neighbours: beyond a wall the mirrored row or column (zero gradient)
  const int xm = x > 0 ? x - 1 : (g.bc_x == BC_WALL ? 0 : g.nx - 1);
  const int xq = x < g.nx - 1 ? x + 1 : (g.bc_x == BC_WALL ? x : 0);
  for (int y = blockIdx.y; y < g.ny; y += gridDim.y) {   // gridDim.y is capped at 65535
    const int ym = y > 0 ? y - 1 : (g.bc_y == BC_WALL ? 0 : g.ny - 1);
    const int yq = y < g.ny - 1 ? y + 1 : (g.bc_y == BC_WALL ? y : 0);
    auto at = [&](int k) { return in.f[k] ? in.f[k][(long long)y * in.pitch[k] + x] : 0.0f; };
    const float *fs = in.f[0] + (long long)ym * in.pitch[0], *fc = in.f[0] + (long long)y * in.pitch[0],
                *fn = in.f[0] + (long long)yq * in.pitch[0];
    const float ph = fc[x], u = at(1), v = at(2), p = at(3);
    // mu0 = theta'(phi0) - kappa lap(phi0) (Eq. 1)
    const float lap =
        (4.0f * (fc[xq] + fn[x] + fc[xm] + fs[x]) + (fn[xq] + fn[xm] + fs[xm] + fs[xq]) - 20.0f * ph) * (1.0f / 6.0f);
    const float m = P.four_beta * ph * (ph * ph - P.phi_star2) - P.kappa * lap;
    const float cl = fminf(fmaxf((ph + P.phi_star) * P.inv_2phistar, 0.0f), 1.0f);
    const float rho = P.rho_B + cl * P.drho;
    const float uu15 = 1.5f * (u * u + v * v);
    char* const dst = static_cast<char*>(g.dst);
    const int row = y * g.row_bytes;
    // the place the value comes from, which keys BF16 rounding: the cell upstream, or the reversed
    // population of the cell itself across a wall
    auto put = [&](auto pop, float val) {
      constexpr int A = decltype(pop)::value;
      constexpr int a = A == A_F0LO ? 0 : A % Q;
      char* q = dst + pop_at<ST>(A, row, cx(a) == 1 ? col.cm : (cx(a) == -1 ? col.cq : col.c0), g);
      if constexpr (pop_bytes(ST, A) == 4) {
        *reinterpret_cast<float*>(q) = val;
      } else {
        int xz = x - cx(a), yz = y - cy(a), from = A;
        const bool hit = (g.bc_x == BC_WALL && (xz < 0 || xz >= g.nx)) || (g.bc_y == BC_WALL && (yz < 0 || yz >= g.ny));
        if (hit) {
          xz = x;
          yz = y;
          from = opp(a) + (A >= Q ? Q : 0);
        }
        *reinterpret_cast<unsigned short*>(q) =
            enc_pop<ST>(to_scale<ST>(P, val), from, hash_key<ST>(wrap1(xz, g.nx), wrap1(yz, g.ny), g));
      }
    };
    float rest = 0.0f;
    auto dir = [&](auto idx) {
      constexpr int a = decltype(idx)::value;
      const float w = wgt(a);
      const float eu = (float)cx(a) * u + (float)cy(a) * v;
      const float poly = 3.0f * eu + 4.5f * eu * eu - uu15;
      put(std::integral_constant<int, Q + a>{}, w * p + rho * (1.0f / 3.0f) * (w * poly));
      if constexpr (a > 0) {
        // f^eq_a: with the mu term, or phi Gamma_a in the forced order-parameter form
        const float feq = w * (P.f_forced ? ph * (1.0f + poly) : P.three_gamma_f * m + ph * poly);
        put(std::integral_constant<int, a>{}, feq);
        rest += feq;
      }
    };
    dir(std::integral_constant<int, 0>{});
    dir(std::integral_constant<int, 1>{});
    dir(std::integral_constant<int, 2>{});
    dir(std::integral_constant<int, 3>{});
    dir(std::integral_constant<int, 4>{});
    dir(std::integral_constant<int, 5>{});
    dir(std::integral_constant<int, 6>{});
    dir(std::integral_constant<int, 7>{});
    dir(std::integral_constant<int, 8>{});
    // f_0^eq = phi - sum_{a>0} f^eq_a, kept as the float pair (hi, lo)
    float hi, lo;
    two_sum(ph, -rest, hi, lo);
    if constexpr (ST == ST_FP32) {
      put(std::integral_constant<int, 0>{}, hi);
      put(std::integral_constant<int, A_F0LO>{}, lo);
    } else {
      put(std::integral_constant<int, 0>{}, hi + lo);
    }
  }
  if (first && stale != 0u) {
    *g.give_up.word = 0u;
    if (g.give_up.host) *static_cast<volatile unsigned int*>(g.give_up.host) = 0u;
  }
}

// s_form 1: rho and div(rho u) of the initial fields, which stand for the step before the first.
__global__ void k_init_sdef(Phys P, Grid g, InitIn in) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.nx) return;
  const int xm = x > 0 ? x - 1 : (g.bc_x == BC_WALL ? 0 : g.nx - 1);
  const int xq = x < g.nx - 1 ? x + 1 : (g.bc_x == BC_WALL ? x : 0);
  for (int y = blockIdx.y; y < g.ny; y += gridDim.y) {   // gridDim.y is capped at 65535
    const int ym = y > 0 ? y - 1 : (g.bc_y == BC_WALL ? 0 : g.ny - 1);
    const int yq = y < g.ny - 1 ? y + 1 : (g.bc_y == BC_WALL ? y : 0);
    auto at = [&](int k, int dx, int dy) {
      const int xx = dx < 0 ? xm : (dx > 0 ? xq : x), yy = dy < 0 ? ym : (dy > 0 ? yq : y);
      return in.f[k] ? in.f[k][(long long)yy * in.pitch[k] + xx] : 0.0f;
    };
    auto rho = [&](int dx, int dy) { return fmad(__saturatef(fmad(at(0, dx, dy), P.inv_2phistar, 0.5f)), P.drho, P.rho_B); };
    auto jx = [&](int dx, int dy) { return fmul(rho(dx, dy), at(1, dx, dy)); };
    auto jy = [&](int dx, int dy) { return fmul(rho(dx, dy), at(2, dx, dy)); };
    const float djx = fmad(4.0f, fsub(jx(1, 0), jx(-1, 0)), fsub(fsub(jx(1, 1), jx(-1, -1)), fsub(jx(-1, 1), jx(1, -1))));
    const float djy = fmad(4.0f, fsub(jy(0, 1), jy(0, -1)), fadd(fsub(jy(1, 1), jy(-1, -1)), fsub(jy(-1, 1), jy(1, -1))));
    float* sp = reinterpret_cast<float*>(static_cast<char*>(g.dst) + g.spoff);
    const long long c = (long long)y * g.pitch + x;
    sp[c] = rho(0, 0);
    sp[g.plane + c] = fmul(fadd(djx, djy), 1.0f / 12.0f);
  }
}

cudaError_t launch_init(const lbm_sim* s, const InitIn& in, cudaStream_t st) {
  Grid g = make_grid(s, nullptr, s->buf[s->cur]);
  dim3 blk(128), grd((s->nx + 127) / 128, s->ny < 65535 ? s->ny : 65535);
  switch (g.storage) {
    case ST_FP16: k_init_pop<ST_FP16><<<grd, blk, 0, st>>>(s->phys, g, in); break;
    case ST_BF16: k_init_pop<ST_BF16><<<grd, blk, 0, st>>>(s->phys, g, in); break;
    default: k_init_pop<ST_FP32><<<grd, blk, 0, st>>>(s->phys, g, in); break;
  }
  if (s->params.s_form) {
    cudaError_t e2 = cudaGetLastError();
    if (e2 != cudaSuccess) return e2;
    k_init_sdef<<<grd, blk, 0, st>>>(s->phys, g, in);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------ checkpoint order
// A checkpoint holds the post-collision populations at their source cells, a row in blocks of 32 cells with
// every population of the block's cells in turn (FP32: f_0..f_8, gbar_0..gbar_8, f_0lo, 128 bytes each;
// 16-bit: the FP32 rest population, then 17 of 64 bytes).  Pad columns keep their place.
//
// A lane moves a cell, or takes two neighbours of 16-bit storage out, whose halves share the checkpoint's words: the
// accesses of a population are 32 neighbouring columns or pairs on both sides, and all populations of a lane are in flight
// together.  4096 x 4096 out / in, us: FP32 392 / 401, 16-bit 258 / 256 (one cell a lane out: 271; two in: 302-335); a copy
// is 405 and 220.  With 16-byte units of the checkpoint, 4 or 8 cells of one population, it was 1003 / 1005 and 1180 / 1150.
template <int... A, class F>
__device__ __forceinline__ void each_pop(std::integer_sequence<int, A...>, F f) {
  (f(std::integral_constant<int, A>{}), ...);
}
constexpr int reorder_cells(int st, bool out) { return st != ST_FP32 && out ? 2 : 1; }
// Groups [k0, k1) of the grid, each the `PER` blocks (fewer at a row's end) that a warp moves; lin: where group 0 would lie.
template <int ST, bool OUT>
__global__ void __launch_bounds__(256) k_reorder(char* __restrict__ state, char* __restrict__ lin, Grid g, long long k0, long long k1) {
  constexpr auto pops = std::make_integer_sequence<int, ST == ST_FP32 ? 19 : 18>{};
  constexpr int BYTES = 32 * (int)state_bytes_per_cell(ST);   // of a block
  constexpr int PER = reorder_cells(ST, OUT);                 // of a lane
  const int groups = (g.nblk + PER - 1) / PER;                // of a row
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long k = k0 + (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5); k < k1; k += warps) {
    const int y = (int)(k / groups), x = (int)(k - (long long)y * groups) * 32 * PER + (threadIdx.x & 31) * PER;
    if (x >= g.pitch) continue;
    char* const part = lin + ((long long)y * g.nblk + (x >> 5)) * BYTES;
    const int at = x & 31;
    auto cell = [&](int xx) {
      OutCell<ST> c = out_cell<ST>(g, xx < g.nx ? xx : 0, y);
      if (xx >= g.nx) {                                       // a pad column: its own place
        c.rm = c.rq = c.r0;
        c.c.c0 = col_bytes<ST>(xx);
        c.wl = c.wr = c.wb = c.wt = false;
      }
      return c;
    };
    const OutCell<ST> c0 = cell(x), c1 = cell(x + PER - 1);
    auto word = [](char* p) -> unsigned int& { return *reinterpret_cast<unsigned int*>(p); };
    auto half = [](char* p) -> unsigned short& { return *reinterpret_cast<unsigned short*>(p); };
    unsigned int v[19];                                       // (16-bit storage: [18] the second rest population)
    each_pop(pops, [&](auto pop) {
      constexpr int A = decltype(pop)::value;
      if constexpr (pop_bytes(ST, A) == 4) {
        v[A] = OUT ? word(state + c0.template at<A>()) : word(part + A * 128 + at * 4);
        if constexpr (PER == 2) v[18] = word(state + c1.template at<A>());
      } else if constexpr (OUT) {
        const unsigned int lo = half(state + c0.template at<A>()), hi = half(state + c1.template at<A>());
        v[A] = lo | hi << 16;
      } else {
        v[A] = half(part + 128 + (A - 1) * 64 + at * 2);
      }
    });
    each_pop(pops, [&](auto pop) {
      constexpr int A = decltype(pop)::value;
      if constexpr (pop_bytes(ST, A) == 4) {
        word(OUT ? part + A * 128 + at * 4 : state + c0.template at<A>()) = v[A];
        if constexpr (PER == 2) word(part + at * 4 + 4) = v[18];
      } else if constexpr (OUT) {
        word(part + 128 + (A - 1) * 64 + at * 2) = v[A];
      } else {
        half(state + c0.template at<A>()) = (unsigned short)v[A];
      }
    });
  }
}

template <int ST>
static cudaError_t launch_reorder_st(const lbm_sim* s, void* state, char* lin, long long k0, long long k1, bool out, cudaStream_t st) {
  const Grid g = make_grid(s, nullptr, nullptr);
  const long long want = (k1 - k0 + 7) / 8;
  const int grid = (int)(want < 64LL * s->sms ? want : 64LL * s->sms);
  char* const first = lin - reorder_offset(s, out, k0);
  if (out) k_reorder<ST, true><<<grid, 256, 0, st>>>(static_cast<char*>(state), first, g, k0, k1);
  else k_reorder<ST, false><<<grid, 256, 0, st>>>(static_cast<char*>(state), first, g, k0, k1);
  return cudaGetLastError();
}

static long long reorder_row(const lbm_sim* s, bool out) {
  const int per = reorder_cells(s->params.storage, out);
  return (s->pitch / BLK + per - 1) / per;
}
long long reorder_groups(const lbm_sim* s, bool out) { return s->ny * reorder_row(s, out); }
long long reorder_offset(const lbm_sim* s, bool out, long long k) {
  const long long row = reorder_row(s, out), per = reorder_cells(s->params.storage, out);
  return ((k / row) * (s->pitch / BLK) + (k % row) * per) * BLK * state_bytes_per_cell(s->params.storage);
}
long long reorder_fit(const lbm_sim* s, bool out, size_t bytes) {
  return (long long)bytes / (reorder_cells(s->params.storage, out) * BLK * state_bytes_per_cell(s->params.storage));
}

cudaError_t launch_reorder(const lbm_sim* s, void* state, void* lin, long long k0, long long k1, bool out, cudaStream_t st) {
  // the two 16-bit storages are laid out alike
  return s->params.storage == LBM_FP32 ? launch_reorder_st<ST_FP32>(s, state, static_cast<char*>(lin), k0, k1, out, st)
                                       : launch_reorder_st<ST_FP16>(s, state, static_cast<char*>(lin), k0, k1, out, st);
}

// ------------------------------------------------------------------ FP64 diagnostics

cudaError_t launch_diag(const lbm_sim* s, cudaStream_t st) {
  const float* f = s->fields;
  double* record = s->slot ? reinterpret_cast<double*>(&s->slot->diag) : s->red + (long long)s->ny * DIAG_PARTIALS;
  const DiagIn d = diag_in(f, f + 2 * s->plane, f + 3 * s->plane, f + 4 * s->plane, s->nx, s->ny, s->pitch, s->phys.phi_star, s->red,
                     record, diag_done(s), s->steps);
  return launch_diag_rows(d, s->sms, st);
}

}  // namespace lbm
