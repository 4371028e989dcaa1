// Ragged batches: many independent simulations (any sizes and parameters) advanced by one
// persistent launch per time step over a work list of (simulation, strip, segment) tiles; one launch per
// storage present, and one more per storage for members that use the direct mass defect.  Steps run as
// replays of one 16-step CUDA graph captured once per membership, the remainder of a step count as direct
// launches.  Each tile runs the row march of the single-simulation kernel (every operation rounded to
// nearest explicitly), so a member's state is bitwise the same alone or inside any mix.
#include <algorithm>
#include <array>
#include <map>
#include <new>
#include <utility>
#include <vector>

#include "lbm_batch.cuh"

using namespace lbm;

constexpr int GRAPH_STEPS = 16;        // steps per captured graph (even: parity-neutral)

constexpr int N_PARTS = 6;              // storage + 3 x (direct mass defect)

struct lbm_batch {
  size_t budget = 0;
  size_t bytes = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t cap = nullptr;          // private stream for graph capture
  std::vector<lbm_sim*> slots;         // nullptr = free slot
  int seg_h = 0;                       // rows per tile for members without their own choice (0: chosen here)
  bool dirty = true;                   // descriptors / work list need rebuilding
  SimDesc* d_sims = nullptr;
  int4* d_work = nullptr;
  unsigned int* d_next = nullptr;      // a tile counter per part
  size_t cap_sims = 0, cap_work = 0;
  int n_work = 0;
  struct Part {                        // tiles of one storage and one form of the mass defect: a launch each
    int first = 0, count = 0, grid = 0, nt = 0;
  } parts[N_PARTS];
  int flip = 0;                        // parity offset of every member since the last rebuild
  bool xwall = true;                   // some member has walls on x (the general kernel form)
  std::map<int, cudaGraphExec_t> graphs;  // flip -> executable graph of GRAPH_STEPS steps
};

static void drop_graphs(lbm_batch* b) {
  for (auto& kv : b->graphs) cudaGraphExecDestroy(kv.second);
  b->graphs.clear();
}

static int rebuild(lbm_batch* b) {
  std::vector<SimDesc> sims;
  std::vector<int4> work;
  std::vector<int> members;
  for (size_t i = 0; i < b->slots.size(); ++i)
    if (b->slots[i]) members.push_back((int)i);
  // members of different storages, and those with the direct mass defect, have launches of their own; a launch
  // takes its tiles in order of falling height
  std::vector<std::pair<int, int4>> per[N_PARTS];
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  b->xwall = false;
  for (int m : members) b->xwall = b->xwall || b->slots[m]->params.bc_x == LBM_WALL;
  auto part_of = [](const lbm_sim* s) { return s->params.storage + (s->params.s_form ? 3 : 0); };
  // Rows per tile.  A launch takes as many rounds as its tiles fill of the device's slots, and a round as many row
  // iterations as its tiles have: the height that makes rounds x (h + 7) least, heights evened out within each member
  // (48 members of the c4 mix, us a step: 171 at the chosen 53 rows, 193 at 56).
  // CTAs of 64 or 32 threads where they save a seventh of that: an iteration takes as long, four or eight CTAs share an
  // SM, and narrow members leave fewer of their threads idle (us a step, FP32: 256 members of
  // 64 x 64 98.5 -> 54.9, 64 of 256 x 256 173.6 -> 138.1, 100 of 33 x 200 101.5 -> 39.3; mixes of 64 to 512 columns stay).
  int rows[N_PARTS], threads[N_PARTS];
  for (int part = 0; part < N_PARTS; ++part) {
    long long best = -1;
    rows[part] = 32;
    threads[part] = MARCH_NT;
    for (int nt = MARCH_NT; nt >= 32; nt /= 2) {
      std::vector<std::array<int, 3>> shape;   // strips, rows, own rows per tile
      bool fits = true;
      for (int m : members) {
        const lbm_sim* s = b->slots[m];
        if (part_of(s) != part) continue;
        const MarchShape q = march_shape_of(s->nx, s->params.storage, s->params.s_form != 0, nt);
        fits = fits && q.strips > 0;
        shape.push_back({q.strips, s->ny, s->seg_h ? s->seg_h : b->seg_h});
      }
      if (!fits || shape.empty()) continue;
      const long long slots = (long long)sms * march_ctas(nt);
      long long least = -1;
      int least_h = 32;
      for (int h = 4; h <= 512; h += h < 64 ? 1 : h / 16) {
        long long tiles = 0;
        for (const auto& q : shape) {
          const int hh = q[2] ? q[2] : h;
          tiles += (long long)q[0] * ((q[1] + hh - 1) / hh);
        }
        const long long cost = (tiles + slots - 1) / slots * (h + 7);
        if (least < 0 || cost < least) {
          least = cost;
          least_h = h;
        }
      }
      if (best < 0 || 7 * least < 6 * best) {
        best = least;
        rows[part] = least_h;
        threads[part] = nt;
      }
    }
  }
  for (size_t m = 0; m < members.size(); ++m) {
    lbm_sim* s = b->slots[members[m]];
    SimDesc d{};
    d.P = s->phys2;
    Grid g = make_grid(s, nullptr, nullptr);
    const int part = part_of(s);
    int h = s->seg_h ? s->seg_h : b->seg_h;
    if (!h) {
      const int segs = (s->ny + rows[part] - 1) / rows[part];
      h = (s->ny + segs - 1) / segs;
    }
    tile_geometry(march_shape_of(s->nx, s->params.storage, s->params.s_form != 0, threads[part]), h, sms, &g);
    g.wait_hold = s->hold;
    d.g = g;
    d.buf0 = s->buf[0];
    d.buf1 = s->buf[1];
    d.cur0 = s->cur;
    sims.push_back(d);
    const int nseg = (s->ny + g.seg_h - 1) / g.seg_h;
    for (int sg = 0; sg < nseg; ++sg) {
      const int tile_rows = std::min(g.seg_h, s->ny - sg * g.seg_h);
      for (int st = 0; st < g.n_strips; ++st) per[part].push_back({tile_rows, make_int4((int)m, st, sg, 0)});
    }
  }
  lbm_batch::Part parts[N_PARTS];
  for (int part = 0; part < N_PARTS; ++part) {
    parts[part].first = (int)work.size();
    std::stable_sort(per[part].begin(), per[part].end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    for (const auto& v : per[part]) work.push_back(v.second);
    parts[part].count = (int)work.size() - parts[part].first;
    parts[part].nt = threads[part];
    parts[part].grid = std::min(parts[part].count, sms * march_ctas(threads[part]));
  }
  cudaError_t e;
  if (sims.size() > b->cap_sims) {
    cudaFree(b->d_sims);
    b->d_sims = nullptr;
    b->cap_sims = 0;
    if ((e = cudaMalloc(&b->d_sims, sims.size() * sizeof(SimDesc))) != cudaSuccess) return cuda_fail(e, "batch descriptors");
    b->cap_sims = sims.size();
  }
  if (work.size() > b->cap_work) {
    cudaFree(b->d_work);
    b->d_work = nullptr;
    b->cap_work = 0;
    if ((e = cudaMalloc(&b->d_work, work.size() * sizeof(int4))) != cudaSuccess) return cuda_fail(e, "batch work list");
    b->cap_work = work.size();
  }
  if (!sims.empty() &&
      (e = cudaMemcpyAsync(b->d_sims, sims.data(), sims.size() * sizeof(SimDesc), cudaMemcpyHostToDevice, b->stream)) !=
          cudaSuccess)
    return cuda_fail(e, "batch descriptor upload");
  if (!work.empty() &&
      (e = cudaMemcpyAsync(b->d_work, work.data(), work.size() * sizeof(int4), cudaMemcpyHostToDevice, b->stream)) !=
          cudaSuccess)
    return cuda_fail(e, "batch work upload");
  if (!b->d_next && (e = cudaMalloc(&b->d_next, N_PARTS * sizeof(unsigned int))) != cudaSuccess)
    return cuda_fail(e, "batch tile counters");
  if ((e = cudaMemsetAsync(b->d_next, 0, N_PARTS * sizeof(unsigned int), b->stream)) != cudaSuccess)
    return cuda_fail(e, "batch tile counters");
  // host vectors die here: make the uploads complete first
  if ((e = cudaStreamSynchronize(b->stream)) != cudaSuccess) return cuda_fail(e, "batch upload sync");
  b->n_work = (int)work.size();
  std::copy(parts, parts + N_PARTS, b->parts);
  b->flip = 0;
  drop_graphs(b);
  b->dirty = false;
  return LBM_OK;
}

// One time step of every member: the launches touch disjoint members.
static cudaError_t launch_batch(lbm_batch* b, int parity, cudaStream_t st) {
  static constexpr decltype(&launch_batch_fp32) by_storage[3] = {launch_batch_fp32, launch_batch_fp16, launch_batch_bf16};
  for (int k = 0; k < N_PARTS; ++k) {
    const lbm_batch::Part& p = b->parts[k];
    if (p.count == 0) continue;
    const BatchPart q{b->d_sims, b->d_work + p.first, p.count, p.grid, parity, p.nt, b->d_next + k, k >= 3, b->xwall};
    const cudaError_t e = by_storage[k % 3](q, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

extern "C" {

int lbm_batch_create(size_t budget_bytes, void* cuda_stream, lbm_batch** out) {
  if (!out) return set_error("out is NULL"), LBM_ERR_INVALID_ARG;
  lbm_batch* b = new (std::nothrow) lbm_batch();
  if (!b) return set_error("host allocation failed"), LBM_ERR_OOM;
  b->budget = budget_bytes;
  b->stream = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    delete b;
    return cuda_fail(e, "batch stream");
  }
  *out = b;
  return LBM_OK;
}

int lbm_batch_add(lbm_batch* b, lbm_sim* s, int* slot) {
  Range range_("lbm_batch_add");
  if (!b || !s) return set_error("batch and sim are required"), LBM_ERR_INVALID_ARG;
  if (s->batch) return set_error("simulation already belongs to a batch"), LBM_ERR_INVALID_ARG;
  if (s->params.f_form)
    return set_error("f_form 1 simulations are stepped alone (the batch kernel has no forced form)"),
           LBM_ERR_INVALID_ARG;
  const size_t need = lbm_sim_device_bytes(s);
  if (b->budget && b->bytes + need > b->budget) {
    set_error("batch budget: %zu + %zu > %zu bytes", b->bytes, need, b->budget);
    return LBM_ERR_BUDGET;
  }
  // the member's earlier work (init, steps) was queued on its own stream
  cudaStreamSynchronize(s->stream);
  int k = -1;
  for (size_t i = 0; i < b->slots.size(); ++i)
    if (!b->slots[i]) {
      k = (int)i;
      break;
    }
  if (k < 0) {
    k = (int)b->slots.size();
    b->slots.push_back(nullptr);
  }
  b->slots[k] = s;
  s->batch = b;
  b->bytes += need;
  b->dirty = true;
  if (slot) *slot = k;
  return LBM_OK;
}

int lbm_batch_remove(lbm_batch* b, int slot) {
  Range range_("lbm_batch_remove");
  if (!b || slot < 0 || slot >= (int)b->slots.size() || !b->slots[slot])
    return set_error("invalid batch slot %d", slot), LBM_ERR_INVALID_ARG;
  lbm_sim* s = b->slots[slot];
  cudaError_t e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "batch remove sync");
  s->batch = nullptr;
  b->bytes -= lbm_sim_device_bytes(s);
  b->slots[slot] = nullptr;
  b->dirty = true;
  return LBM_OK;
}

int lbm_batch_step(lbm_batch* b, int k) {
  Range range_("lbm_batch_step");
  if (!b || k < 0) return set_error("invalid batch or step count"), LBM_ERR_INVALID_ARG;
  if (k == 0) return LBM_OK;
  int rc;
  if (b->dirty && (rc = rebuild(b))) return rc;
  if (b->n_work == 0) return LBM_OK;
  // Whole blocks of GRAPH_STEPS steps replay one graph captured once per membership (the block
  // is even, so a replay leaves the buffer parity as it found it); the remaining k mod
  // GRAPH_STEPS steps are launched directly.  Round lengths then vary freely without a new
  // capture each time.
  const int blocks = k / GRAPH_STEPS, rest = k % GRAPH_STEPS;
  cudaError_t e = cudaSuccess;
  if (blocks > 0) {
    cudaGraphExec_t exec = nullptr;
    auto it = b->graphs.find(b->flip);
    if (it != b->graphs.end()) {
      exec = it->second;
    } else {
      cudaGraph_t graph;
      e = cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) return cuda_fail(e, "batch capture begin");
      for (int i = 0; i < GRAPH_STEPS && e == cudaSuccess; ++i) e = launch_batch(b, b->flip + i, b->cap);
      cudaError_t e2 = cudaStreamEndCapture(b->cap, &graph);
      if (e != cudaSuccess) return cuda_fail(e, "batch capture launch");
      if (e2 != cudaSuccess) return cuda_fail(e2, "batch capture end");
      e = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return cuda_fail(e, "batch graph instantiate");
      b->graphs[b->flip] = exec;
    }
    for (int i = 0; i < blocks && e == cudaSuccess; ++i) e = cudaGraphLaunch(exec, b->stream);
    if (e != cudaSuccess) return cuda_fail(e, "batch graph launch");
  }
  for (int i = 0; i < rest && e == cudaSuccess; ++i) e = launch_batch(b, b->flip + i, b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "batch step launch");
  bool flip = (k & 1) != 0;
  for (lbm_sim* s : b->slots) {
    if (!s) continue;
    s->steps += k;
    s->launches += k;
    if (flip) s->cur ^= 1;
  }
  if (flip) b->flip ^= 1;
  return LBM_OK;
}

int lbm_batch_set_tile(lbm_batch* b, int threads, int seg_rows) {
  if (!b) return set_error("batch is NULL"), LBM_ERR_INVALID_ARG;
  if (threads && threads != 64 && threads != 128 && threads != 256)
    return set_error("threads must be 64, 128 or 256"), LBM_ERR_INVALID_ARG;
  if (seg_rows < 0) return set_error("seg_rows must be >= 1"), LBM_ERR_INVALID_ARG;
  if (seg_rows) b->seg_h = seg_rows;
  b->dirty = true;
  return LBM_OK;
}

int lbm_batch_set_tile_auto(lbm_batch* b) {
  if (!b) return set_error("batch is NULL"), LBM_ERR_INVALID_ARG;
  b->seg_h = 0;
  b->dirty = true;
  return LBM_OK;
}

int lbm_batch_size(const lbm_batch* b) {
  if (!b) return 0;
  int n = 0;
  for (lbm_sim* s : b->slots) n += s != nullptr;
  return n;
}

size_t lbm_batch_bytes(const lbm_batch* b) { return b ? b->bytes : 0; }

int lbm_batch_destroy(lbm_batch* b) {
  if (!b) return LBM_OK;
  cudaStreamSynchronize(b->stream);
  for (lbm_sim* s : b->slots)
    if (s) s->batch = nullptr;
  drop_graphs(b);
  cudaFree(b->d_sims);
  cudaFree(b->d_work);
  cudaFree(b->d_next);
  if (b->cap) cudaStreamDestroy(b->cap);
  delete b;
  return LBM_OK;
}

}  // extern "C"
