// The row march: the fused step (and the moment evaluation) of a simulation whose grid fills the
// device, for every configuration.
//
// A CTA marches up a strip of columns and a segment of rows [ya, yb).  Each thread owns two columns, one
// in each half ("lane") of the strip: thread t has the columns x0 - 3 + t and x0 + w - 3 + t, w columns per
// lane plus a 3-column halo on each side (march_shape in lbm_api.cu has the choice of threads and strips).  Every value is a V2, the pair of the two lanes, so one
// packed instruction, one 64-bit shared-memory access and one address serve two cells.
//
// Row iteration a runs four stages in two phases, a barrier after each:
//   phase 1   S0  row a     phi = sum_a f_a
//             S2  row a-3   grad phi, grad mu, lap mu, rho, F_s, G, s, u, p        [Eq. 4, 5, 8]
//   phase 2   S1  row a-1   mu = theta'(phi) - kappa lap(phi)                      [Eq. 1]
//             S3  row a-4   grad p, grad psi, div u, both collisions, stores
// The two stages of a phase do not depend on each other and read only what earlier phases wrote, so they
// are one stretch of independent work for the scheduler.  Their stencils work on rings of rows in
// shared memory; a segment of h rows takes h + 7 iterations.
//
// The populations come into shared memory by bulk copies (cp.async.bulk), one per region for the row's whole
// chunk of columns (two where a strip wraps around the edge of a periodic grid), STAGES rows ahead.  They
// hold neither registers nor L1 lines while in flight.
//
// Why this form (2048 x 512 and 4096 x 4096, FP32 storage): the step moves 152 B per cell, 6.5 cycles
// per cell and SM at the measured bandwidth.  With one cell per thread it issued 594-745 warp instructions per
// 32 cells, 4.6-5.8 cycles per cell at best, and its warps waited 30-48 % of their time on loads that one row of
// register prefetch could not cover (more warps or L2 prefetches only thrashed L1).  This form issues 380 per 32 cells.
// 4096 x 4096: 527 -> 408 us a step (152 B per cell at 0.92 of the measured copy bandwidth); 2048 x 512 with walls on y:
// 40.8 -> 32.4, of which 1.5 us pass between two launches, 5.3 in the iterations before a segment's first S3 (1.4 of
// them for the first row), 1.4 in each of the others.  What bounds an iteration is a warp's own chain of about 760
// instructions at 4.3 cycles (2 warps per scheduler; issue slots half used, shared-memory pipe 65 %): warps that skip
// columns beyond the halo, or more rows in flight, change nothing.
#pragma once
#include "lbm_device.cuh"

namespace lbm {

enum { MODE_STEP = 0, MODE_MOMENTS = 1 };

// Threads per CTA (NT): 128, 64 or 32, and 2, 4 or 8 such CTAs per SM (shared memory; 8 warps of up to 255 registers).
constexpr int MARCH_NT = 128;
__host__ __device__ constexpr int march_ctas(int nt) { return 256 / nt; }
// Blocks of a staged row.  128 threads: what any strip of 2 x 122 columns can touch (s_form 1: one less, so that its
// additional rings fit).  64: as many as let four CTAs share an SM.  32: whole rows of up to 52 columns only.
__host__ __device__ constexpr int march_slots(int nt, int st, bool sd) {
  return nt == 128 ? (sd ? 9 : 10) : (nt == 32 ? 2 : (st == ST_FP32 ? (sd ? 4 : 5) : 6));
}
// The blocks of columns that a strip of w columns per lane at x0 stages: [b0, b0 + run1) and, where it wraps, [0, run2).
struct StagedRun {
  int b0, run1, run2;
};
__host__ __device__ __forceinline__ StagedRun staged_run(int nx, int x0, int w) {
  const int nbx = (nx + BLK - 1) / BLK;
  if (nx < 2 * w + 8) return StagedRun{0, nbx, 0};
  const int xs = wrap1(x0 - 4, nx), xe = wrap1(x0 + 2 * w + 3, nx), b0 = xs / BLK;
  return xs <= xe ? StagedRun{b0, xe / BLK - b0 + 1, 0} : StagedRun{b0, nbx - b0, xe / BLK + 1};
}
constexpr int STAGES = 2;                 // rows of f and of gbar in shared memory or in flight
constexpr int RING5 = 5;                  // rows a-4 .. a of phi and of the f populations awaiting S3
constexpr int RING3 = 3;                  // rows of mu, p, u

template <int ST, bool SD, int NT>
struct MarchSmem {
  static constexpr int NSLOT = march_slots(NT, ST, SD);
  struct Stage {                          // 16-byte aligned pieces
    unsigned char f[NSLOT * region_block(ST, R_F)], l[NSLOT * region_block(ST, R_L)], g[NSLOT * region_block(ST, R_G)];
  };
  struct Row5 {
    ulonglong2 f[4][NT];                  // f_1..f_8 of both lanes, own column
    V2 hi[NT], lo[NT];
  };
  struct Row3 {
    V2 mu[NT], p[NT], ux[NT], uy[NT];
    V2 j[SD ? 2 : 0][NT];                 // rho u (direct mass defect)
  };
  alignas(128) unsigned long long fbar[STAGES];
  unsigned long long gbar[STAGES];
  unsigned int quit;                      // a wait of this CTA ran out
  int2 left[2];                           // where its producers of f and of gbar then stopped (StageAt)
  alignas(128) Stage stage[STAGES];
  Row5 r5[RING5];
  Row3 r3[RING3];
  V2 tail[2];                             // the last thread reads one column past its ring row
};

__device__ __forceinline__ unsigned int smem_u32(const void* p) { return (unsigned int)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* b, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(unsigned int dst, const void* src, int bytes, unsigned long long* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(b))
               : "memory");
}
// True once the phase `parity` of a barrier has completed (after a short wait in the instruction itself).
__device__ __forceinline__ bool mbar_try(unsigned long long* b, int parity) {
  unsigned int done;
  asm volatile("{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(done)
               : "r"(smem_u32(b)), "r"(parity)
               : "memory");
  return done != 0;
}

// Before the first tile of a CTA.
template <int ST, bool SD, int NT>
__device__ __forceinline__ void march_init(MarchSmem<ST, SD, NT>& sm) {
  if (threadIdx.x == 0) {
    for (int k = 0; k < STAGES; ++k) {
      mbar_init(&sm.fbar[k]);
      mbar_init(&sm.gbar[k]);
    }
    sm.quit = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// Store where `on`, as one predicated instruction: no branch around it.
__device__ __forceinline__ void st_on(float* p, float v, bool on) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q st.global.f32 [%0], %1;\n\t}" ::"l"(p), "f"(v),
               "r"((int)on));
}

// The two lanes' new populations, and the store of one lane's: the gbar (and the f) populations together under
// one predicate, to the rows they stream to.
template <int ST>
struct OutLanes {
  mutable V2 v[Q + Q + 1];
  template <int A>
  __device__ __forceinline__ void put(V2 x) const {
    v[A] = x;
  }
  template <bool B>
  __device__ __forceinline__ void lane(float x[Q + Q + 1]) const {
#pragma unroll
    for (int a = 0; a < (ST == ST_FP32 ? 19 : 18); ++a) {
      float lo, hi;
      unpack2(v[a], lo, hi);
      x[a] = B ? hi : lo;
    }
  }
  // rows: the destination buffer's rows y-1, y, y+1; x: the lane's column; key: its BF16 rounding place.  wb, wt: the row
  // lies at the bottom or the top wall (uniform); XW: the column may lie at the left (wl) or the right (wr) wall.  The
  // populations that would cross a wall go back reversed: to row y, column x + e_x (wrapped).  (Storing all
  // populations of such a cell by tests of their own instead took a row body for the segments at walls on y, cold code
  // that few CTAs ran: a step after a flush of L2 42 us against 37 on 2048 x 512; and with walls on x 39.5 against 37.6
  // on 1200 x 900.)
  template <bool B, bool XW>
  __device__ __forceinline__ void store_lane(const Grid& gr, char* rm, char* r0, char* rq, int x_, unsigned int key, bool on, bool wl,
                                             bool wr, bool wb, bool wt) const {
    float x[Q + Q + 1];
    lane<B>(x);
    const int nblk = gr.nblk;
    const ColB c = col_bytes<ST>(x_);
    const int right = on && !(XW && wr), left = on && !(XW && wl);
    const int up = on && !wt, down = on && !wb, up_r = right && !wt, up_l = left && !wt, down_r = right && !wb, down_l = left && !wb;
    const int g = region_start(ST, R_G) * nblk + c.g;
    static_assert(BLK == 32, "offsets below");
    if constexpr (ST == ST_FP32) {
      asm volatile(
          "{\n\t.reg .pred q, r, l, t, tr, tl, b, br, bl;\n\tsetp.ne.s32 q, %0, 0;\n\tsetp.ne.s32 r, %13, 0;\n\tsetp.ne.s32 l, %14, 0;\n\t"
          "setp.ne.s32 t, %15, 0;\n\tsetp.ne.s32 tr, %16, 0;\n\tsetp.ne.s32 tl, %17, 0;\n\tsetp.ne.s32 b, %18, 0;\n\t"
          "setp.ne.s32 br, %19, 0;\n\tsetp.ne.s32 bl, %20, 0;\n\t"
          "@t st.global.f32 [%1+256], %4;\n\t@tr st.global.f32 [%1+640], %5;\n\t@tl st.global.f32 [%1+768], %6;\n\t"
          "@q st.global.f32 [%2], %7;\n\t@r st.global.f32 [%2+128], %8;\n\t@l st.global.f32 [%2+384], %9;\n\t"
          "@b st.global.f32 [%3+512], %10;\n\t@bl st.global.f32 [%3+896], %11;\n\t@br st.global.f32 [%3+1024], %12;\n\t}" ::"r"(
              (int)on),
          "l"(rq + g), "l"(r0 + g), "l"(rm + g), "f"(x[Q + 2]), "f"(x[Q + 5]), "f"(x[Q + 6]), "f"(x[Q + 0]), "f"(x[Q + 1]),
          "f"(x[Q + 3]), "f"(x[Q + 4]), "f"(x[Q + 7]), "f"(x[Q + 8]), "r"(right), "r"(left), "r"(up), "r"(up_r), "r"(up_l),
          "r"(down), "r"(down_r), "r"(down_l));
      asm volatile(
          "{\n\t.reg .pred q, r, l, t, tr, tl, b, br, bl;\n\tsetp.ne.s32 q, %0, 0;\n\tsetp.ne.s32 r, %15, 0;\n\tsetp.ne.s32 l, %16, 0;\n\t"
          "setp.ne.s32 t, %17, 0;\n\tsetp.ne.s32 tr, %18, 0;\n\tsetp.ne.s32 tl, %19, 0;\n\tsetp.ne.s32 b, %20, 0;\n\t"
          "setp.ne.s32 br, %21, 0;\n\tsetp.ne.s32 bl, %22, 0;\n\t"
          "@t st.global.f32 [%1+256], %5;\n\t@tr st.global.f32 [%1+640], %6;\n\t@tl st.global.f32 [%1+768], %7;\n\t"
          "@q st.global.f32 [%2], %8;\n\t@r st.global.f32 [%2+128], %9;\n\t@l st.global.f32 [%2+384], %10;\n\t"
          "@b st.global.f32 [%3+512], %11;\n\t@bl st.global.f32 [%3+896], %12;\n\t@br st.global.f32 [%3+1024], %13;\n\t"
          "@q st.global.f32 [%4], %14;\n\t}" ::"r"((int)on),
          "l"(rq + c.f4), "l"(r0 + c.f4), "l"(rm + c.f4), "l"(r0 + region_start(ST, R_L) * nblk + c.l), "f"(x[2]), "f"(x[5]),
          "f"(x[6]), "f"(x[0]), "f"(x[1]), "f"(x[3]), "f"(x[4]), "f"(x[7]), "f"(x[8]), "f"(x[A_F0LO]), "r"(right), "r"(left), "r"(up), "r"(up_r), "r"(up_l),
          "r"(down), "r"(down_r), "r"(down_l));
      if (wl || wr || wb || wt) back<XW>(gr, r0, x_, on, wl, wr, wb, wt, [&](auto a) { return x[decltype(a)::value]; });
    } else {
      unsigned short h[Q + Q];
#pragma unroll
      for (int a = 1; a < (ST == ST_BF16 ? Q : Q + Q); ++a) h[a] = enc_pop<ST>(x[a], a, key);
      if constexpr (ST == ST_BF16) {               // gbar: two per conversion
#pragma unroll
        for (int a = Q; a < Q + Q - 1; a += 2) {
          const unsigned int d = bf16_stochastic2(x[a], key + pop_key(a), x[a + 1], key + pop_key(a + 1));
          h[a] = static_cast<unsigned short>(d);
          h[a + 1] = static_cast<unsigned short>(d >> 16);
        }
        h[Q + Q - 1] = enc_pop<ST>(x[Q + Q - 1], Q + Q - 1, key);
      }
      asm volatile(
          "{\n\t.reg .pred q, r, l, t, tr, tl, b, br, bl;\n\tsetp.ne.s32 q, %0, 0;\n\tsetp.ne.s32 r, %13, 0;\n\tsetp.ne.s32 l, %14, 0;\n\t"
          "setp.ne.s32 t, %15, 0;\n\tsetp.ne.s32 tr, %16, 0;\n\tsetp.ne.s32 tl, %17, 0;\n\tsetp.ne.s32 b, %18, 0;\n\t"
          "setp.ne.s32 br, %19, 0;\n\tsetp.ne.s32 bl, %20, 0;\n\t"
          "@t st.global.u16 [%1+128], %4;\n\t@tr st.global.u16 [%1+320], %5;\n\t@tl st.global.u16 [%1+384], %6;\n\t"
          "@q st.global.u16 [%2], %7;\n\t@r st.global.u16 [%2+64], %8;\n\t@l st.global.u16 [%2+192], %9;\n\t"
          "@b st.global.u16 [%3+256], %10;\n\t@bl st.global.u16 [%3+448], %11;\n\t@br st.global.u16 [%3+512], %12;\n\t}" ::"r"(
              (int)on),
          "l"(rq + g), "l"(r0 + g), "l"(rm + g), "h"(h[Q + 2]), "h"(h[Q + 5]), "h"(h[Q + 6]), "h"(h[Q + 0]), "h"(h[Q + 1]),
          "h"(h[Q + 3]), "h"(h[Q + 4]), "h"(h[Q + 7]), "h"(h[Q + 8]), "r"(right), "r"(left), "r"(up), "r"(up_r), "r"(up_l),
          "r"(down), "r"(down_r), "r"(down_l));
      asm volatile(
          "{\n\t.reg .pred q, r, l, t, tr, tl, b, br, bl;\n\tsetp.ne.s32 q, %0, 0;\n\tsetp.ne.s32 r, %14, 0;\n\tsetp.ne.s32 l, %15, 0;\n\t"
          "setp.ne.s32 t, %16, 0;\n\tsetp.ne.s32 tr, %17, 0;\n\tsetp.ne.s32 tl, %18, 0;\n\tsetp.ne.s32 b, %19, 0;\n\t"
          "setp.ne.s32 br, %20, 0;\n\tsetp.ne.s32 bl, %21, 0;\n\t"
          "@t st.global.u16 [%1+192], %5;\n\t@tr st.global.u16 [%1+384], %6;\n\t@tl st.global.u16 [%1+448], %7;\n\t"
          "@r st.global.u16 [%2+128], %8;\n\t@l st.global.u16 [%2+256], %9;\n\t"
          "@b st.global.u16 [%3+320], %10;\n\t@bl st.global.u16 [%3+512], %11;\n\t@br st.global.u16 [%3+576], %12;\n\t"
          "@q st.global.f32 [%4], %13;\n\t}" ::"r"((int)on),
          "l"(rq + c.f2), "l"(r0 + c.f2), "l"(rm + c.f2), "l"(r0 + c.f4), "h"(h[2]), "h"(h[5]), "h"(h[6]), "h"(h[1]), "h"(h[3]),
          "h"(h[4]), "h"(h[7]), "h"(h[8]), "f"(x[0]), "r"(right), "r"(left), "r"(up), "r"(up_r), "r"(up_l),
          "r"(down), "r"(down_r), "r"(down_l));
      if (wl || wr || wb || wt) back<XW>(gr, r0, x_, on, wl, wr, wb, wt, [&](auto a) { return h[decltype(a)::value]; });
    }
  }

  // The populations that cross a wall, from value(a).
  template <bool XW, class F>
  __device__ __forceinline__ static void back(const Grid& g, char* r0, int x, bool on, bool wl, bool wr, bool wb, bool wt, F value) {
    const ColB c = col_bytes<ST>(x), cq = col_bytes<ST>(x == g.nx - 1 ? 0 : x + 1), cm = col_bytes<ST>(x == 0 ? g.nx - 1 : x - 1);
    // population first ? A : opp(A), to the reversed population at column to
    auto put = [&](auto pop, bool first, const ColB& to) {
      constexpr int A = decltype(pop)::value, M = opp(A % Q) + (A >= Q ? Q : 0);
      char* const q = r0 + region_start(ST, region_of(A)) * g.nblk + (first ? pop_in_region<ST>(M, to) : pop_in_region<ST>(A, to));
      const auto v = first ? value(std::integral_constant<int, A>{}) : value(std::integral_constant<int, M>{});
      if (on) *reinterpret_cast<std::remove_const_t<decltype(v)>*>(q) = v;
    };
    if (wb || wt) {
      put(std::integral_constant<int, 2>{}, wt, c);
      put(std::integral_constant<int, 5>{}, wt, wt ? cq : cm);
      put(std::integral_constant<int, 6>{}, wt, wt ? cm : cq);
      put(std::integral_constant<int, Q + 2>{}, wt, c);
      put(std::integral_constant<int, Q + 5>{}, wt, wt ? cq : cm);
      put(std::integral_constant<int, Q + 6>{}, wt, wt ? cm : cq);
    }
    if (XW && (wl || wr)) {
      const ColB& cw = wr ? cq : cm;
      put(std::integral_constant<int, 1>{}, wr, cw);
      put(std::integral_constant<int, 5>{}, wr, cw);
      put(std::integral_constant<int, 8>{}, wr, cw);
      put(std::integral_constant<int, Q + 1>{}, wr, cw);
      put(std::integral_constant<int, Q + 5>{}, wr, cw);
      put(std::integral_constant<int, Q + 8>{}, wr, cw);
    }
  }
};

// One row iteration (kinds).  Rows at a wall on y have no kind of their own: their stencils take the row itself for the
// one beyond it, and their stores turn back what crosses the wall.  (A third, checked body for segments at a wall: 228
// instead of 208 registers, spills in the batch, and those segments the slowest: 2048 x 512 FP32 35.0 us a step against
// 32.4, FP16 33.2 against 29.4; 900 x 300 14.6 against 13.1; 48 batched members BF16 187 against 171.)
//   IT_FILL     the first iterations of a segment: no S3 yet, S2 from its first needed row on.
//   IT_INNER    all stages.
// Threads whose column a stage does not need compute it anyway, from whatever the rings hold;
// only stores to the new state (and, with walls on x, to the rings) are predicated.
enum { IT_FILL = 1, IT_INNER = 2 };

// The stage the next row of f (or gbar) is read from, and the parity of its barrier.
struct StageAt {
  int stage = 0, parity = 0;
  __device__ __forceinline__ void next() {
    if (++stage == STAGES) {
      stage = 0;
      parity ^= 1;
    }
  }
  __device__ __forceinline__ int ahead(int k) const { return stage + k >= STAGES ? stage + k - STAGES : stage + k; }
};

// SD: the direct mass defect (s_form 1) is compiled in.  FF: the forced order-parameter LBE (f_form 1;
// FP32 storage only).  XW: the x axis may have walls.  K: the scheme constants (Phys2, in the constant bank
// or in shared memory).
// PDL: the launch is a programmatic dependent of the previous one and waits for it here, once its addresses are formed.
// give_up: in the constant bank or in global memory, read when a wait runs out: the tile is then left undone, sm.quit is
// set, and the CTA must not march again.
template <int MODE, int ST, bool SD, bool FF, bool XW, bool PDL, int NT, class K>
__device__ __forceinline__ void march(const K& P, const Grid& g, const GiveUp* give_up, const MomentOut& mo, int strip, int seg,
                                      MarchSmem<ST, SD, NT>& sm, StageAt& fat, StageAt& gat) {
  constexpr int GT = NT > 32 ? 32 : 16;            // the thread that copies gbar (thread 0 copies f)
  const int t = threadIdx.x;
  const int w = g.tile_w;
  const int x0 = strip * 2 * w;
  const int wa = min(w, g.nx - x0), wb = min(w, g.nx - x0 - w);   // columns of each lane (wb may be < 1)
  const int ya = seg * g.seg_h;
  const int yb = min(ya + g.seg_h, g.ny);
  const int te = min(t, w + 5);                    // threads beyond the halo repeat its last column
  const int xla = x0 - 3 + te, xlb = xla + w;      // logical columns (may lie outside [0, nx))
  const int xpa = wrap1(xla, g.nx), xpb = wrap1(xlb, g.nx);
  const bool on_a = t >= 3 && t < wa + 3, on_b = t >= 3 && t < wb + 3;
  const bool ywall = g.bc_y == BC_WALL;

  // ---- staged columns
  const StagedRun run = staged_run(g.nx, x0, w);
  const int b0 = run.b0, run1 = run.run1, run2 = run.run2;
  auto staged_col = [&](int xp) {
    const int blk = xp / BLK;
    return col_bytes<ST>(blk >= b0 ? blk - b0 : run1 + blk, xp & (BLK - 1));
  };
  auto staged3 = [&](int xp) {
    return Col3{staged_col(xp == 0 ? g.nx - 1 : xp - 1), staged_col(xp), staged_col(xp == g.nx - 1 ? 0 : xp + 1)};
  };
  const Col3 ca = staged3(xpa), cb = staged3(xpb);
  // x walls: the columns next to one, and the ghost column their threads also fill
  const bool xwall = XW && g.bc_x == BC_WALL;
  const bool real_a = !xwall || (xla >= 0 && xla < g.nx), real_b = !xwall || (xlb >= 0 && xlb < g.nx);
  auto ghost_of = [&](int xl) {
    if (!xwall || t != te) return -1;
    return xl == 0 ? t - 1 : (xl == g.nx - 1 && t + 1 < NT ? t + 1 : -1);
  };
  const int tga = ghost_of(xla), tgb = ghost_of(xlb);

  // ---- producer: one thread copies the rows of f, another (of another warp, if there is one) those of gbar
  auto load_piece = [&](unsigned char* dst, int r, int region, unsigned long long* bar) {
    const int blk = region_block(ST, region);
    const char* row = static_cast<const char*>(g.src) + (long long)wrap1(r, g.ny) * g.row_bytes + region_start(ST, region) * g.nblk;
    bulk_load(smem_u32(dst), row + b0 * blk, run1 * blk, bar);
    if (run2 > 0) bulk_load(smem_u32(dst) + run1 * blk, row, run2 * blk, bar);
  };
  int role = t;                            // 0, GT: producer; -1 once a wait of this thread has run out
  // rows fr of f into stage fs and gr of gbar into stage gs
  auto produce = [&](bool do_f, int fr, int fs, bool do_g, int gr, int gs) {
    if (role == 0 && do_f) {
      mbar_expect(&sm.fbar[fs], (run1 + run2) * (region_block(ST, R_F) + region_block(ST, R_L)));
      load_piece(sm.stage[fs].f, fr, R_F, &sm.fbar[fs]);
      if constexpr (region_block(ST, R_L) > 0) load_piece(sm.stage[fs].l, fr, R_L, &sm.fbar[fs]);
    }
    if (role == GT && do_g) {
      mbar_expect(&sm.gbar[gs], (run1 + run2) * region_block(ST, R_G));
      load_piece(sm.stage[gs].g, gr, R_G, &sm.gbar[gs]);
    }
  };

  // S2 runs in iterations ya + 2 .. a_end (rows ya - 1 ..), S3 in ya + 4 .. yb + 3; the moment pass ends
  // with S2 of row yb - 1.
  const int a_end = MODE == MODE_STEP ? yb + 3 : yb + 2;
  if constexpr (PDL) {
    // until the previous grid has completed and its stores are visible; then let the next launch proceed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  const bool held = MODE == MODE_STEP && g.wait_hold == seg * g.n_strips + strip;
  for (int k = 0; k < STAGES; ++k)
    produce(!held, ya - 3 + k, fat.ahead(k), !held && ya - 1 + k <= a_end - 3, ya - 1 + k, gat.ahead(k));

  // ---- rings: byte offsets of this thread's place in the rows a-k (mod 5) and a-k (mod 3) of iteration a.  The
  // rows of mu (read a-4 .. a-2, then a-1 written) and of p, u (a-3 written, then a-5 .. a-3 read) share
  // the second set.
  using S = MarchSmem<ST, SD, NT>;
  char* const base = reinterpret_cast<char*>(&sm);
  int q5[RING5], q3[RING3];
#pragma unroll
  for (int k = 0; k < RING5; ++k) q5[k] = (int)offsetof(S, r5) + (RING5 - 1 - k) * (int)sizeof(typename S::Row5) + t * 8;
#pragma unroll
  for (int k = 0; k < RING3; ++k) q3[k] = (int)offsetof(S, r3) + (RING3 - 1 - k) * (int)sizeof(typename S::Row3) + t * 8;
  auto at = [&](int off) { return reinterpret_cast<V2*>(base + off); };
  constexpr int HI = offsetof(typename S::Row5, hi), LO = offsetof(typename S::Row5, lo);
  constexpr int MU = offsetof(typename S::Row3, mu), PP = offsetof(typename S::Row3, p), UX = offsetof(typename S::Row3, ux),
                UY = offsetof(typename S::Row3, uy), JX = offsetof(typename S::Row3, j), JY = JX + 8 * NT;
  // The lanes whose column is real store it, and next to a wall on x also its mirror image in the ghost column.
  // Threads away from the walls store both lanes at once.
  const bool plain = !XW || (real_a && real_b && tga < 0 && tgb < 0);
  auto put_wall = [&](int off, V2 v) {
    float x, y;
    unpack2(v, x, y);
    float* const f = reinterpret_cast<float*>(at(off));
    if (real_a) f[0] = x;
    if (real_b) f[1] = y;
    if (tga >= 0) f[2 * (tga - t)] = x;
    if (tgb >= 0) f[2 * (tgb - t) + 1] = y;
  };
  auto put = [&](int off, V2 v) { *at(off) = v; };
  // Offsets of the rows south and north of row r.  Beyond a wall they are the row itself, its mirror image.  (The rows
  // beyond it go through the stages too, from the wrapped rows of the grid: no valid row reads what they leave.)
  const int wall_lo = ywall ? 0 : -8, wall_hi = ywall ? g.ny - 1 : g.ny + 8;
  auto south = [&](int r, int s, int c) { return r == wall_lo ? c : s; };
  auto north = [&](int r, int n, int c) { return r == wall_hi ? c : n; };

  // ---- population pop of both lanes from a staged region
  auto staged = [&](const unsigned char* reg, auto pop, const ColB& a, const ColB& b) {
    constexpr int A = decltype(pop)::value;
    auto one = [&](const ColB& c) {
      const unsigned char* q = reg + pop_in_region<ST>(A, c);
      if constexpr (pop_bytes(ST, A) == 4) return *reinterpret_cast<const float*>(q);
      else return dec_pop<ST>(*reinterpret_cast<const unsigned short*>(q), A);
    };
    return pack2(one(a), one(b));
  };
  // the populations F .. F + 8 that stream into the lanes' cells
  auto pull9 = [&](auto first, const unsigned char* reg, V2 v[Q]) {
    constexpr int F = decltype(first)::value;
    v[0] = staged(reg, std::integral_constant<int, F + 0>{}, ca.c0, cb.c0);
    v[1] = staged(reg, std::integral_constant<int, F + 1>{}, ca.cm, cb.cm);
    v[2] = staged(reg, std::integral_constant<int, F + 2>{}, ca.c0, cb.c0);
    v[3] = staged(reg, std::integral_constant<int, F + 3>{}, ca.cq, cb.cq);
    v[4] = staged(reg, std::integral_constant<int, F + 4>{}, ca.c0, cb.c0);
    v[5] = staged(reg, std::integral_constant<int, F + 5>{}, ca.cm, cb.cm);
    v[6] = staged(reg, std::integral_constant<int, F + 6>{}, ca.cq, cb.cq);
    v[7] = staged(reg, std::integral_constant<int, F + 7>{}, ca.cq, cb.cq);
    v[8] = staged(reg, std::integral_constant<int, F + 8>{}, ca.cm, cb.cm);
  };
  using F0 = std::integral_constant<int, 0>;
  using G0 = std::integral_constant<int, Q>;

  RecT<V2> cur{}, prev{};                  // records of rows a-3 and a-4 (in phase 2 of iteration a)
  V2 gcur[Q], gprev[Q];                    // their pulled gbar
  // phi and 12 grad(phi) as S1 meets them, for S2 two iterations later: rows a-2 and a-3 in phase 1 of iteration a
  struct PhiGrad {
    V2 ph, gx, gy;
  } pg2{}, pg3{};
  // Direct mass defect: rho, div(rho u) of the last step, read an iteration ahead.  Scalars, packed where they are used:
  // packed at the load they were waited for there (32 x 65536 402 -> 331 us a step, 1000 x 701 33.1 -> 28.7; FP16 as before).
  float sp_ra = 0.0f, sp_rb = 0.0f, sp_da = 0.0f, sp_db = 0.0f;
  auto fetch_sd = [&](int r) {
    if constexpr (SD) {
      const float* sp = reinterpret_cast<const float*>(static_cast<const char*>(g.src) + g.spoff) + wrap1(r, g.ny) * g.pitch;
      sp_ra = __ldg(sp + xpa);
      sp_rb = __ldg(sp + xpb);
      sp_da = __ldg(sp + g.plane + xpa);
      sp_db = __ldg(sp + g.plane + xpb);
    }
  };

  auto shift = [&] {
    prev = cur;
#pragma unroll
    for (int k = 0; k < Q; ++k) gprev[k] = gcur[k];
  };

  // Wait for a staged row, a counted number of tries.  Past that the thread waits no more and copies no more, and what is
  // left of the tile runs through on what the rings hold, so that the iterations need no test of their own.  (With one
  // and a way out of the loop, or with a clock in the wait: 2048 x 512 FP16 5-7 % slower, 601 x 437 with x walls 6-10 %.)
  int tries = g.wait_tries;
  auto wait_row = [&](unsigned long long* b, int parity) {
    for (int n = 0; n < tries; ++n)
      if (mbar_try(b, parity)) return;
    if (role == 0) sm.left[0] = make_int2(fat.stage, fat.parity);
    if (role == GT) sm.left[1] = make_int2(gat.stage, gat.parity);
    tries = 1;
    role = -1;
    sm.quit = 1u;
    give_up->raise();
  };

  auto iter = [&](int a, auto kind) {
    constexpr int KIND = decltype(kind)::value;
    constexpr bool IN = KIND == IT_INNER;
    const int fs = fat.stage, gs = gat.stage;
    const int r1 = a - 1, r2 = a - 3, r3 = a - 4;   // rows of S1, S2, S3
    const bool s2_runs = IN || a >= ya + 2;
    // ================ phase 1: S0 and S2; all stores to the rings at its end
    wait_row(&sm.fbar[fs], fat.parity);
    if (s2_runs) wait_row(&sm.gbar[gs], gat.parity);
    // ---- S0: phi at row a (as an unevaluated pair hi + lo)
    V2 fp[NF], hi, lo;
    auto stage0 = [&] {
      pull9(F0{}, sm.stage[fs].f, fp);
      fp[Q] = zero<V2>();
      if constexpr (ST == ST_FP32) fp[Q] = staged(sm.stage[fs].l, std::integral_constant<int, A_F0LO>{}, ca.c0, cb.c0);
      phi_pair<ST>(P, fp, hi, lo);
    };
    // ---- S2: u, p at row a-3 (rows a-4 .. a-2 of phi and mu)
    S2Out<V2> o;
    auto stage2 = [&] {
      const int c3 = q3[0], s3 = south(r2, q3[1], c3), n3 = north(r2, q3[2], c3);
      const V2 *ms = at(s3 + MU), *m0 = at(c3 + MU), *mn = at(n3 + MU);
      const V2 ph = pg3.ph, gphx = pg3.gx, gphy = pg3.gy;
      V2 gmx, gmy;                                 // 12 x the isotropic gradient
      grad12(P, ms, m0, mn, gmx, gmy);
      V2 sdef;
      if constexpr (SD) sdef = fadd(fsub(density(P, ph), pack2(sp_ra, sp_rb)), pack2(sp_da, sp_db));
      else sdef = fmul(P.s_coef6, lap6_of(P, ms, m0, mn));
      asm("" : "+l"(sdef.v));                      // computed either way: no branch around the stencil
      [[maybe_unused]] const V2 s_all = sdef;      // F_a is reported whether or not the scheme removes it
      sdef.v = P.remove_Fa ? sdef.v : 0ull;
      V2 gb[Q];
      pull9(G0{}, sm.stage[gs].g, gb);
      o = s2_cell<ST>(P, ph, gphx, gphy, gmx, gmy, m0[0], sdef, gb);
      if constexpr (MODE == MODE_STEP) {
        if constexpr (SD) {
          float x, y;                              // rho^t for the next step
          unpack2(o.rho, x, y);
          float* sp = reinterpret_cast<float*>(static_cast<char*>(g.dst) + g.spoff) + (long long)r2 * g.pitch;
          const bool row = r2 >= ya && r2 < yb;
          st_on(sp + xpa, x, on_a && row);
          st_on(sp + xpb, y, on_b && row);
        }
        shift();
        s2_record(P, o, ph, m0[0], sdef, cur);
#pragma unroll
        for (int k = 0; k < Q; ++k) gcur[k] = gb[k];
        if constexpr (FF) {
          cur.gx12 = gphx;
          cur.gy12 = gphy;
          cur.lmu6 = lap6_of(P, ms, m0, mn);
        }
      } else if (r2 >= ya) {                       // r2 < yb throughout
        auto store2 = [&](float* q, V2 v) {
          float x, y;
          unpack2(v, x, y);
          if (on_a) q[r2 * mo.pitch + xpa] = x;
          if (on_b) q[r2 * mo.pitch + xpb] = y;
        };
        if (mo.phi) store2(mo.phi, ph);
        if (mo.rho) store2(mo.rho, o.rho);
        if (mo.ux) store2(mo.ux, o.ux);
        if (mo.uy) store2(mo.uy, o.uy);
        if (mo.p) store2(mo.p, o.p);
        if (mo.fax) {
          store2(mo.fax, fmul(fsub(zero<V2>(), o.ux), s_all));
          store2(mo.fay, fmul(fsub(zero<V2>(), o.uy), s_all));
        }
      }
    };
    stage0();
    if (s2_runs) stage2();
    auto puts1 = [&](auto put_) {
      put_(q5[0] + HI, hi);
      put_(q5[0] + LO, lo);
      if (s2_runs) {
        put_(q3[0] + PP, o.p);
        if constexpr (MODE == MODE_STEP) {
          put_(q3[0] + UX, o.ux);
          put_(q3[0] + UY, o.uy);
          if constexpr (SD) {
            put_(q3[0] + JX, fmul(o.rho, o.ux));
            put_(q3[0] + JY, fmul(o.rho, o.uy));
          }
        }
      }
    };
    if (!XW || plain) puts1(put);
    else puts1(put_wall);
    if (MODE == MODE_STEP) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        *reinterpret_cast<ulonglong2*>(base + q5[0] + t * 8 + k * NT * 16) = make_ulonglong2(fp[2 * k + 1].v, fp[2 * k + 2].v);
    }
    if (IN || a >= ya + 1) fetch_sd(r2 + 1);
    __syncthreads();
    // ================ phase 2: S1 and S3
    // the stages just read are free
    produce(a + STAGES <= a_end, a + STAGES, fs, s2_runs && r2 + STAGES <= a_end - 3, r2 + STAGES, gs);
    // ---- S1: mu at row a-1 (rows a-2 .. a of phi)
    V2 mu;
    auto stage1 = [&] {
      const int c = q5[1], sr = south(r1, q5[2], c), n = north(r1, q5[0], c);
      mu = chem_potential(P, at(sr + HI), at(c + HI), at(n + HI), at(sr + LO), at(c + LO), at(n + LO));
      // grad phi only feeds grad rho (density and pressure terms): the high words suffice
      pg2.ph = fadd(*at(c + HI), *at(c + LO));
      grad12(P, at(sr + HI), at(c + HI), at(n + HI), pg2.gx, pg2.gy);
    };
    // ---- S3: collide and store row a-4 (p, u of rows a-5 .. a-3)
    auto stage3 = [&] {
      const int c = q3[1], os = south(r3, q3[2], c), on = north(r3, q3[0], c);
      V2 gpx, gpy;                                 // 12 grad p
      grad12(P, at(os + PP), at(c + PP), at(on + PP), gpx, gpy);
      // phi div(u) of the convective form; computed either way, so that no branch splits the block
      V2 phiD = phi_div_u(P, prev.phi, at(os + UX), at(c + UX), at(on + UX), at(os + UY), at(on + UY));
      asm("" : "+l"(phiD.v));
      phiD.v = P.ch_conv ? phiD.v : 0ull;
      V2 f[Q];
      f[0] = zero<V2>();   // unused: f_0 follows from the phi pair
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(base + q5[4] + t * 8 + k * NT * 16);
        f[2 * k + 1].v = v.x;
        f[2 * k + 2].v = v.y;
      }
      if constexpr (SD) {
        // div(rho u) of this step, for the next step's mass defect
        const V2 *xs = at(os + JX), *xc = at(c + JX), *xn = at(on + JX), *ys = at(os + JY), *yn = at(on + JY);
        const V2 djx = fmad(P.k4, fsub(xc[1], xc[-1]), fsub(fsub(xn[1], xs[-1]), fsub(xn[-1], xs[1])));
        const V2 djy = fmad(P.k4, fsub(yn[0], ys[0]), fadd(fsub(yn[1], ys[-1]), fsub(yn[-1], ys[1])));
        float x, y;
        unpack2(fmul(fadd(djx, djy), P.k12th), x, y);
        float* sp = reinterpret_cast<float*>(static_cast<char*>(g.dst) + g.spoff) + g.plane + (long long)r3 * g.pitch;
        st_on(sp + xpa, x, on_a);
        st_on(sp + xpb, y, on_b);
      }
      OutLanes<ST> out;
      collide_store<ST, FF>(P, prev, *at(c + PP), gpx, gpy, *at(q5[4] + HI), *at(q5[4] + LO), phiD, f, gprev, out);
      char* const dst = static_cast<char*>(g.dst);
      char* const row0 = dst + (long long)r3 * g.row_bytes;
      char* const rowm = r3 == 0 ? dst + (long long)(g.ny - 1) * g.row_bytes : row0 - g.row_bytes;
      char* const rowq = r3 == g.ny - 1 ? dst : row0 + g.row_bytes;
      const bool wb = r3 == wall_lo, wt = r3 == wall_hi;
      out.template store_lane<false, XW>(g, rowm, row0, rowq, xpa, hash_key<ST>(xpa, r3, g), on_a, xwall && xla == 0,
                                         xwall && xla == g.nx - 1, wb, wt);
      out.template store_lane<true, XW>(g, rowm, row0, rowq, xpb, hash_key<ST>(xpb, r3, g), on_b, xwall && xlb == 0,
                                        xwall && xlb == g.nx - 1, wb, wt);
    };
    pg3 = pg2;
    stage1();
    if constexpr (MODE == MODE_STEP && IN) stage3();
    if (!XW || plain) put(q3[1] + MU, mu);
    else put_wall(q3[1] + MU, mu);
    {
      const int x5 = q5[RING5 - 1], x3 = q3[RING3 - 1];
#pragma unroll
      for (int k = RING5 - 1; k > 0; --k) q5[k] = q5[k - 1];
#pragma unroll
      for (int k = RING3 - 1; k > 0; --k) q3[k] = q3[k - 1];
      q5[0] = x5;
      q3[0] = x3;
    }
    fat.next();
    if (s2_runs) gat.next();
    __syncthreads();
  };

  using Fill = std::integral_constant<int, IT_FILL>;
  using Inner = std::integral_constant<int, IT_INNER>;
  int a = ya - 3;
  for (; a < ya + 4 && a <= a_end; ++a) iter(a, Fill{});
  for (; a <= a_end; ++a) iter(a, Inner{});
  // A tile that was given up: copies in flight write to this CTA's shared memory, so their producer waits for them, as
  // long again.
  if (sm.quit != 0u) {
    if (role != t && (t == 0 || t == GT)) {
      unsigned long long* const bar = t == 0 ? sm.fbar : sm.gbar;
      StageAt at;
      at.stage = sm.left[t != 0].x;
      at.parity = sm.left[t != 0].y;
      int n = 0;
      for (int k = 0; k < STAGES; ++k, at.next())
        while (n < g.wait_tries && !mbar_try(bar + at.stage, at.parity)) ++n;
    }
    __syncthreads();
  }
}

}  // namespace lbm
