// lb_batch.cu -- many independent domains stepped together.
//
// Contexts of the fused scheme are grouped into classes that share one
// compiled brick shape (lattice, storage, brick, pipeline) and the forcing
// switch.  Per time step each class runs ONE persistent launch: a grid of as
// many CTAs as fit on the GPU at once, each sweeping a fixed slice of a work
// list that holds every brick column of every domain of the class.  The list
// is balanced once, on the host, by greedy longest-processing-time assignment
// of the bricks (cost = nodes x planes incl. pipeline fill) to the CTAs.  The
// launches of two consecutive steps of all classes are captured in a CUDA
// graph and replayed, so a long run costs one graph launch per two steps.
//
// In calls of several steps, members of some size run one by one on a few
// streams of the batch in moment form (lb_k3.cuh, lb_k4.cu), side by side and beside the classes of
// the members that are left: a second list of classes and a second graph.
//
// The per-node arithmetic, the bricks and the shells are exactly those of
// the domain's own single-domain launches: every domain's populations are bit
// for bit those of stepping it alone.
#include <algorithm>
#include <cstring>
#include <new>
#include <queue>
#include <vector>

#include "lb_k1_launch.cuh"

struct lb_batch {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<lb_ctx*> ctxs;
  struct Class {
    const lbgb::K1Variant* v = nullptr;
    bool force = false;
    std::vector<int> members;  // indices into ctxs
    void* d_args = nullptr;    // K1Args<R>[2][n]
    CUtensorMap* d_tmaps = nullptr;
    int4* d_items = nullptr;
    int* d_starts = nullptr;
    int* d_par = nullptr;
    int* h_par = nullptr;  // pinned mirror of d_par
    int n_items = 0, grid = 0;
  };
  std::vector<Class> classes;
  std::vector<int> runs;    // members that calls of several steps run on their own,
  std::vector<int> lane;    // the stream (of lanes) that each of them runs on, and
  std::vector<Class> rest;  // the classes of the others
  int* d_status = nullptr;
  cudaGraphExec_t graph = nullptr;       // two steps of all classes, and
  cudaGraphExec_t rest_graph = nullptr;  // of the rest
  cudaEvent_t done = nullptr;
  cudaEvent_t fork = nullptr;          // class branches of one step
  std::vector<cudaStream_t> side;      // one per class after the first
  std::vector<cudaEvent_t> join;
  std::vector<cudaEvent_t> ctx_ev;
  std::vector<cudaStream_t> lanes;
  std::vector<cudaEvent_t> lane_ev;
  int64_t steps_done = 0;
  int64_t total_nodes = 0;
  double* d_sums = nullptr;  // lb_batch_reduce: seven sums per member (device)
  double* h_sums = nullptr;  // and their pinned host copy
};

namespace lbgb {
namespace {

int cuda_rc(cudaError_t e) { return e == cudaSuccess ? LB_OK : (e == cudaErrorMemoryAllocation ? LB_E_NOMEM : LB_E_CUDA); }

#define LB_BTRY(x)                      \
  do {                                  \
    cudaError_t e_ = (x);               \
    if (e_ != cudaSuccess) return cuda_rc(e_); \
  } while (0)

struct DevGuard {
  int prev = -1;
  explicit DevGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (dev >= 0 && dev != prev) cudaSetDevice(dev);
  }
  ~DevGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

void free_class(lb_batch::Class& c) {
  if (c.d_args) cudaFree(c.d_args);
  if (c.d_tmaps) cudaFree(c.d_tmaps);
  if (c.d_items) cudaFree(c.d_items);
  if (c.d_starts) cudaFree(c.d_starts);
  if (c.d_par) cudaFree(c.d_par);
  if (c.h_par) cudaFreeHost(c.h_par);
  c = lb_batch::Class{};
}

// Static balance: bricks by decreasing cost, each to the least-loaded CTA.
// A brick costs its full cross-section times its planes plus the pipeline
// fill: the warps of a ragged brick issue for their idle lanes too.
void build_work_list(const lb_batch& b, const lb_batch::Class& c, int grid, std::vector<int4>& items,
                     std::vector<int>& starts) {
  struct Brick {
    double cost;
    int4 it;
  };
  std::vector<Brick> all;
  for (int m = 0; m < int(c.members.size()); ++m) {
    const lb_ctx* x = b.ctxs[c.members[m]];
    const FusedPlan& p = x->plan;
    for (int k = 0; k < p.nbz; ++k)
      for (int j = 0; j < p.nby; ++j)
        for (int i = 0; i < p.nbx; ++i) {
          const int bz = std::min(p.bz, x->g.nz - k * p.bz);
          all.push_back({double(p.bx) * p.by * (bz + p.slots + 2), make_int4(m, i, j, k)});
        }
  }
  std::stable_sort(all.begin(), all.end(), [](const Brick& a, const Brick& b2) { return a.cost > b2.cost; });
  using Load = std::pair<double, int>;
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
  for (int g = 0; g < grid; ++g) heap.push({0.0, g});
  std::vector<std::vector<int4>> per(grid);
  for (const Brick& br : all) {
    Load l = heap.top();
    heap.pop();
    per[l.second].push_back(br.it);
    l.first += br.cost;
    heap.push(l);
  }
  items.clear();
  starts.assign(grid + 1, 0);
  for (int g = 0; g < grid; ++g) {
    starts[g] = int(items.size());
    items.insert(items.end(), per[g].begin(), per[g].end());
  }
  starts[grid] = int(items.size());
}

int setup_class(lb_batch& b, lb_batch::Class& c) {
  const int n = int(c.members.size());
  const int occ = c.v->batched_occupancy();
  if (occ <= 0) return LB_E_CUDA;
  std::vector<int4> items;
  std::vector<int> starts;
  int64_t bricks = 0;
  for (int m : c.members) {
    const FusedPlan& p = b.ctxs[m]->plan;
    bricks += int64_t(p.nbx) * p.nby * p.nbz;
  }
  const int grid = int(std::min<int64_t>(bricks, int64_t(k1_sm_count()) * occ));
  build_work_list(b, c, grid, items, starts);
  c.grid = grid;
  c.n_items = int(items.size());
  // arguments of every member at both shell parities, pointing at the batch's status word
  const bool dbl = b.ctxs[c.members[0]]->real_bytes == 8;
  std::vector<K1Args<float>> argsf;
  std::vector<K1Args<double>> argsd;
  (dbl ? argsd.resize(2 * size_t(n)) : argsf.resize(2 * size_t(n)));
  std::vector<CUtensorMap> maps(n);
  for (int m = 0; m < n; ++m) {
    lb_ctx* x = b.ctxs[c.members[m]];
    for (int p = 0; p < 2; ++p) {
      if (dbl) {
        K1Args<double> a = k1_make_args<double>(x, p, 1 - p);
        dispatch_lattice(x->lattice, [&](auto Lt) { make_bounce_terms<decltype(Lt), double>(x->g, a.bb); });
        a.status = b.d_status;
        argsd[size_t(p) * n + m] = a;
      } else {
        K1Args<float> a = k1_make_args<float>(x, p, 1 - p);
        dispatch_lattice(x->lattice, [&](auto Lt) { make_bounce_terms<decltype(Lt), float>(x->g, a.bb); });
        a.status = b.d_status;
        argsf[size_t(p) * n + m] = a;
      }
    }
    maps[m] = x->tmap;
  }
  const size_t args_bytes = dbl ? argsd.size() * sizeof(K1Args<double>) : argsf.size() * sizeof(K1Args<float>);
  const void* args_src = dbl ? static_cast<const void*>(argsd.data()) : static_cast<const void*>(argsf.data());
  LB_BTRY(cudaMalloc(&c.d_args, args_bytes));
  LB_BTRY(cudaMalloc(reinterpret_cast<void**>(&c.d_tmaps), maps.size() * sizeof(CUtensorMap)));
  LB_BTRY(cudaMalloc(reinterpret_cast<void**>(&c.d_items), std::max<size_t>(1, items.size()) * sizeof(int4)));
  LB_BTRY(cudaMalloc(reinterpret_cast<void**>(&c.d_starts), starts.size() * sizeof(int)));
  LB_BTRY(cudaMalloc(reinterpret_cast<void**>(&c.d_par), n * sizeof(int)));
  LB_BTRY(cudaHostAlloc(reinterpret_cast<void**>(&c.h_par), n * sizeof(int), cudaHostAllocDefault));
  LB_BTRY(cudaMemcpyAsync(c.d_args, args_src, args_bytes, cudaMemcpyHostToDevice, b.stream));
  LB_BTRY(cudaMemcpyAsync(c.d_tmaps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice,
                          b.stream));
  if (!items.empty())
    LB_BTRY(cudaMemcpyAsync(c.d_items, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice, b.stream));
  LB_BTRY(cudaMemcpyAsync(c.d_starts, starts.data(), starts.size() * sizeof(int), cudaMemcpyHostToDevice, b.stream));
  for (int m = 0; m < n; ++m) c.h_par[m] = -1;  // forces an upload before the first step
  return LB_OK;
}

// The brick that a batch gives a member: the first plain compiled shape (in
// the planner's order) whose bricks pad the cross-section by at most 25 %, else
// the least padded one; and, for sweeps of up to 256 planes, one brick per
// column, so that small domains do not pay the pipeline fill (slots + 2
// planes) and the z-shell of short bricks (bz; 0: the planner's choice).
const K1Variant* batch_variant(const Geometry& g, int storage, int* bz) {
  const void* vs[64];
  const int nv = std::min(k1_variants_for(g.lattice, storage, vs, 64), 64);
  const K1Variant* pick = nullptr;
  const K1Variant* least = nullptr;
  double least_waste = 1e300;
  for (int i = 0; i < nv; ++i) {
    const K1Variant* v = static_cast<const K1Variant*>(vs[i]);
    // plain shapes only: the decoupled-export and TMA-store alternatives
    // measure slower on the large domains they were tried on
    if (!v->batched || v->nxw != 0 || v->ts != 0) continue;
    const double px = double((g.nx + v->bx - 1) / v->bx) * v->bx;
    const double py = double((g.ny + v->by - 1) / v->by) * v->by;
    const double waste = px * py / (double(g.nx) * double(g.ny));
    if (!pick && waste <= 1.25) pick = v;
    if (waste < least_waste) {
      least_waste = waste;
      least = v;
    }
  }
  *bz = g.nz <= 256 ? g.nz : 0;
  return pick ? pick : least;
}

// Re-plan a member for batched throughput.  Bits are unchanged.
int batch_replan(lb_ctx* x) {
  int bz = 0;
  const K1Variant* pick = batch_variant(x->g, x->storage, &bz);
  FusedPlan want;
  if (!pick || !k1_plan_variant(x->g, pick, bz, &want)) return LB_E_UNSUPPORTED;
  if (pick == k1_ctx_variant(x) && want.bz == x->plan.bz) return LB_OK;
  return ctx_replan(x, pick, bz);
}

constexpr int kShortestSplit = 64;  // planes

// Split the bricks of a class that would not give each of its persistent
// CTAs at least two: halving its members' sweep length (down to kShortestSplit planes)
// doubles their bricks, so that the static work list balances, at the price
// of one more pipeline fill (slots + 2 planes) per added brick.  Bits are
// unchanged.
int split_for_balance(lb_batch& b, lb_batch::Class& c) {
  const int occ = c.v->batched_occupancy();
  if (occ <= 0) return LB_E_CUDA;
  const int64_t cap = int64_t(k1_sm_count()) * occ;
  for (int round = 0; round < 8; ++round) {
    int64_t bricks = 0;
    for (int m : c.members) {
      const FusedPlan& p = b.ctxs[m]->plan;
      bricks += int64_t(p.nbx) * p.nby * p.nbz;
    }
    if (bricks >= 2 * cap) return LB_OK;
    bool changed = false;
    for (int m : c.members) {
      lb_ctx* x = b.ctxs[m];
      if (x->plan.bz <= kShortestSplit) continue;
      const int rc = ctx_replan(x, c.v, std::max(kShortestSplit, (x->plan.bz + 1) / 2));
      if (rc != LB_OK) return rc;
      changed = true;
    }
    if (!changed) return LB_OK;
  }
  return LB_OK;
}

// The members that calls of several steps run on their own, the largest first:
// as many as keep kMeanRunNodes on average, a 2D node counting for 2.5 (its runs
// take several steps per launch).  A step of such a run costs the host about a
// microsecond and the device a launch of few bricks, which the members together
// have to be worth; the classes carry many small ones at less.  100 steps, classes
// against runs: 24 D3Q19 members of 48^3 11.7 / 12.6 ms, 48 D2Q9 members of 300^2
// 12.3 / 3.6, 24 mixed members of 17^3 to 115^3 and 36^2 to 958^2 41 / 17.
std::vector<int> runs_alone(const std::vector<lb_ctx*>& ctxs) {
  constexpr double kMeanRunNodes = 160 * 1024;
  std::vector<int> order(ctxs.size()), runs;
  for (size_t i = 0; i < order.size(); ++i) order[i] = int(i);
  auto weight = [&](int i) { return double(ctxs[i]->n_nodes) * (ctxs[i]->g.d == 2 ? 2.5 : 1.0); };
  std::stable_sort(order.begin(), order.end(), [&](int i, int j) { return weight(i) > weight(j); });
  double sum = 0.0;
  for (int i : order) {
    if (sum + weight(i) < kMeanRunNodes * double(runs.size() + 1)) break;
    if (!moment_plan(ctxs[i]) && !flat_plan(ctxs[i])) continue;
    sum += weight(i);
    runs.push_back(i);
  }
  return runs;
}

// One step (k = 0 or 1 of the captured pair) of every class.  Classes are
// independent domains: each runs on its own branch (the batch stream for the
// first, a side stream forked from it for the others) and all join back.
int launch_classes(lb_batch& b, std::vector<lb_batch::Class>& classes, int k) {
  const int nc = int(classes.size());
  if (nc > 1) {
    LB_BTRY(cudaEventRecord(b.fork, b.stream));
    for (int i = 1; i < nc; ++i) LB_BTRY(cudaStreamWaitEvent(b.side[i - 1], b.fork, 0));
  }
  for (int i = 0; i < nc; ++i) {
    auto& c = classes[i];
    const BatchLaunch L{c.d_args, int(c.members.size()), c.d_tmaps, c.d_items, c.d_starts, c.d_par,
                        c.grid, k, c.force};
    LB_BTRY(c.v->batched(L, i == 0 ? b.stream : b.side[i - 1]));
  }
  for (int i = 1; i < nc; ++i) {
    LB_BTRY(cudaEventRecord(b.join[i - 1], b.side[i - 1]));
    LB_BTRY(cudaStreamWaitEvent(b.stream, b.join[i - 1], 0));
  }
  return LB_OK;
}

// upload each member's current shell parity if it changed since the last step
int sync_parities(lb_batch& b, std::vector<lb_batch::Class>& classes) {
  for (auto& c : classes) {
    bool changed = false;
    for (size_t m = 0; m < c.members.size(); ++m) {
      const int p = b.ctxs[c.members[m]]->parity;
      if (c.h_par[m] != p) changed = true;
    }
    if (!changed) continue;
    // the previous upload may still be in flight: wait before rewriting the pinned mirror
    LB_BTRY(cudaStreamSynchronize(b.stream));
    for (size_t m = 0; m < c.members.size(); ++m) c.h_par[m] = b.ctxs[c.members[m]]->parity;
    LB_BTRY(cudaMemcpyAsync(c.d_par, c.h_par, c.members.size() * sizeof(int), cudaMemcpyHostToDevice, b.stream));
  }
  return LB_OK;
}

// two consecutive steps of the classes as a graph
int capture_pair(lb_batch& b, std::vector<lb_batch::Class>& classes, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  LB_BTRY(cudaStreamBeginCapture(b.stream, cudaStreamCaptureModeThreadLocal));
  int rc = launch_classes(b, classes, 0);
  if (rc == LB_OK) rc = launch_classes(b, classes, 1);
  const cudaError_t e = cudaStreamEndCapture(b.stream, &g);
  if (rc == LB_OK) rc = cuda_rc(e);
  if (rc == LB_OK) rc = cuda_rc(cudaGraphInstantiate(out, g, 0));
  if (g) cudaGraphDestroy(g);
  return rc;
}

// n steps of the given classes on the batch stream
int step_classes(lb_batch& b, std::vector<lb_batch::Class>& classes, cudaGraphExec_t graph, int64_t n) {
  int rc = sync_parities(b, classes);
  if (rc != LB_OK) return rc;
  for (int64_t s = 0; s + 1 < n; s += 2) LB_BTRY(cudaGraphLaunch(graph, b.stream));
  if (n & 1) rc = launch_classes(b, classes, 0);
  if (rc != LB_OK) return rc;
  for (auto& c : classes)
    for (int m : c.members) {
      if (n & 1) b.ctxs[m]->parity = 1 - b.ctxs[m]->parity;
      b.ctxs[m]->steps_done += n;
    }
  return LB_OK;
}

}  // namespace

size_t batch_shell_bytes(const Geometry& g, int storage, size_t room) {
  const size_t real_bytes = storage == LB_F64 ? 8 : 4;
  int bz = 0;
  const K1Variant* v = batch_variant(g, storage, &bz);
  FusedPlan p;
  if (!v || !k1_plan_variant(g, v, bz, &p)) return 0;
  // as many bricks as split_for_balance() may make of a column
  for (size_t most = 0;; p.bz = std::max(kShortestSplit, (p.bz + 1) / 2)) {
    if (!k1_plan_variant(g, v, p.bz, &p)) return most;
    const size_t bytes = size_t(2) * size_t(p.parity_elems) * real_bytes;
    if (bytes > room) most = std::max(most, bytes);
    if (p.bz <= kShortestSplit) return most;
  }
}

}  // namespace lbgb

using namespace lbgb;

extern "C" {

int lb_batch_create(lb_ctx* const* ctxs, int32_t n, void* stream, lb_batch** out) {
  if (!out || !ctxs || n < 1) return LB_E_INVAL;
  *out = nullptr;
  const int dev = ctxs[0] ? ctxs[0]->device : -1;
  for (int i = 0; i < n; ++i) {
    lb_ctx* x = ctxs[i];
    if (!x || x->device != dev) return LB_E_INVAL;
    if (x->scheme != LB_SCHEME_FUSED) return LB_E_UNSUPPORTED;
    // a slab bordering others steps between halo exchanges, not in a batch
    if (x->g.zlink[0] || x->g.zlink[1]) return LB_E_UNSUPPORTED;
    for (int j = 0; j < i; ++j)
      if (ctxs[j] == x) return LB_E_INVAL;
    const K1Variant* v = k1_ctx_variant(x);
    if (!v || !v->batched) return LB_E_UNSUPPORTED;
  }
  DevGuard guard(dev);
  lb_batch* b = new (std::nothrow) lb_batch();
  if (!b) return LB_E_NOMEM;
  b->device = dev;
  int rc = LB_OK;
  do {
    if (stream) {
      b->stream = static_cast<cudaStream_t>(stream);
    } else {
      if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) { rc = LB_E_CUDA; break; }
      b->own_stream = true;
    }
    b->ctxs.assign(ctxs, ctxs + n);
    for (int i = 0; i < n && rc == LB_OK; ++i) {
      // the domain's own stream must be done before the batch reads its state
      if (cudaStreamSynchronize(ctxs[i]->stream) != cudaSuccess) rc = LB_E_CUDA;
      else rc = batch_replan(ctxs[i]);
    }
    if (rc != LB_OK) break;
    for (int i = 0; i < n; ++i) {
      lb_ctx* x = ctxs[i];
      b->total_nodes += x->n_nodes;
      const K1Variant* v = k1_ctx_variant(x);
      const bool force = x->g.has_force;
      auto it = std::find_if(b->classes.begin(), b->classes.end(),
                             [&](const lb_batch::Class& c) { return c.v == v && c.force == force; });
      if (it == b->classes.end()) {
        b->classes.emplace_back();
        b->classes.back().v = v;
        b->classes.back().force = force;
        it = b->classes.end() - 1;
      }
      it->members.push_back(i);
    }
    if (rc != LB_OK) break;
    for (auto& c : b->classes) {
      rc = split_for_balance(*b, c);
      if (rc != LB_OK) break;
    }
    if (rc != LB_OK) break;
    if (cudaMalloc(reinterpret_cast<void**>(&b->d_status), sizeof(int)) != cudaSuccess) { rc = LB_E_NOMEM; break; }
    if (cudaMemsetAsync(b->d_status, 0, sizeof(int), b->stream) != cudaSuccess) { rc = LB_E_CUDA; break; }
    for (auto& c : b->classes) {
      rc = setup_class(*b, c);
      if (rc != LB_OK) break;
    }
    if (rc != LB_OK) break;
    if (cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming) != cudaSuccess) { rc = LB_E_CUDA; break; }
    if (cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess) { rc = LB_E_CUDA; break; }
    for (size_t i = 1; i < b->classes.size() && rc == LB_OK; ++i) {
      cudaStream_t st = nullptr;
      cudaEvent_t ev = nullptr;
      if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) rc = LB_E_CUDA;
      else b->side.push_back(st);
      if (rc == LB_OK && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) rc = LB_E_CUDA;
      else if (rc == LB_OK) b->join.push_back(ev);
    }
    if (rc != LB_OK) break;
    b->ctx_ev.resize(n, nullptr);
    for (int i = 0; i < n && rc == LB_OK; ++i)
      if (cudaEventCreateWithFlags(&b->ctx_ev[i], cudaEventDisableTiming) != cudaSuccess) rc = LB_E_CUDA;
    if (rc != LB_OK) break;
    if ((rc = capture_pair(*b, b->classes, &b->graph)) != LB_OK) break;
    // members that run alone, and the classes without them
    b->runs = runs_alone(b->ctxs);
    // (eight lanes: the streams that the device runs side by side by default),
    // each to the least loaded
    const size_t lanes = std::min<size_t>(b->runs.size(), 8);
    std::vector<int64_t> load(lanes, 0);
    for (int i : b->runs) {
      const size_t k = std::min_element(load.begin(), load.end()) - load.begin();
      b->lane.push_back(int(k));
      load[k] += ctxs[i]->n_nodes;
    }
    for (size_t k = 0; k < lanes && rc == LB_OK; ++k) {
      cudaStream_t st = nullptr;
      cudaEvent_t ev = nullptr;
      rc = cuda_rc(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
      if (rc == LB_OK) b->lanes.push_back(st);
      if (rc == LB_OK) rc = cuda_rc(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
      if (rc == LB_OK) b->lane_ev.push_back(ev);
    }
    if (rc != LB_OK) break;
    if (!b->runs.empty()) {
      for (const auto& c : b->classes) {
        lb_batch::Class r;
        r.v = c.v;
        r.force = c.force;
        for (int m : c.members)
          if (std::find(b->runs.begin(), b->runs.end(), m) == b->runs.end()) r.members.push_back(m);
        if (r.members.empty()) continue;
        b->rest.push_back(r);
        if ((rc = setup_class(*b, b->rest.back())) != LB_OK) break;
      }
      if (rc == LB_OK && !b->rest.empty()) rc = capture_pair(*b, b->rest, &b->rest_graph);
      if (rc != LB_OK) break;
    }
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) { rc = LB_E_CUDA; break; }
  } while (false);
  if (rc != LB_OK) {
    lb_batch_destroy(b);
    return rc;
  }
  *out = b;
  return LB_OK;
}

int lb_batch_step(lb_batch* b, int64_t n) {
  if (!b || n < 0) return LB_E_INVAL;
  if (n == 0) return LB_OK;
  DevGuard guard(b->device);
  // order after work queued on the members' own streams
  for (size_t i = 0; i < b->ctxs.size(); ++i) {
    LB_BTRY(cudaEventRecord(b->ctx_ev[i], b->ctxs[i]->stream));
    LB_BTRY(cudaStreamWaitEvent(b->stream, b->ctx_ev[i], 0));
  }
  int rc = LB_OK;
  if (n >= kMomentMinSteps && !b->runs.empty()) {
    LB_BTRY(cudaEventRecord(b->done, b->stream));
    for (cudaStream_t st : b->lanes)
      if (rc == LB_OK) rc = cuda_rc(cudaStreamWaitEvent(st, b->done, 0));
    for (size_t k = 0; k < b->runs.size() && rc == LB_OK; ++k) {
      lb_ctx* x = b->ctxs[b->runs[k]];
      // the launches of a run go to the stream of the context
      const cudaStream_t own = x->stream;
      x->stream = b->lanes[b->lane[k]];
      rc = cuda_rc(x->g.d == 3 ? moment_run_beside(x, n) : flat_run(x, n, true));
      x->stream = own;
    }
    if (rc == LB_OK && !b->rest.empty()) rc = step_classes(*b, b->rest, b->rest_graph, n);
    // the batch stream waits for what the lanes were given, also where a later
    // launch failed: nothing may run behind the caller's back
    for (size_t k = 0; k < b->lanes.size(); ++k) {
      cudaError_t e = cudaEventRecord(b->lane_ev[k], b->lanes[k]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->lane_ev[k], 0);
      if (rc == LB_OK) rc = cuda_rc(e);
    }
    if (rc == LB_OK)
      for (int i : b->runs) b->ctxs[i]->steps_done += n;
  } else {
    rc = step_classes(*b, b->classes, b->graph, n);
  }
  // later work on a member's stream sees the batch's steps
  cudaError_t e = cudaEventRecord(b->done, b->stream);
  for (lb_ctx* x : b->ctxs)
    if (e == cudaSuccess) e = cudaStreamWaitEvent(x->stream, b->done, 0);
  if (rc == LB_OK) rc = cuda_rc(e);
  if (rc == LB_OK) b->steps_done += n;
  return rc;
}

int lb_batch_sync(lb_batch* b) {
  if (!b) return LB_E_INVAL;
  DevGuard guard(b->device);
  int st = 0;
  LB_BTRY(cudaMemcpyAsync(&st, b->d_status, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
  // members that ran alone report to their own status word
  std::vector<int> own(b->runs.size(), 0);
  for (size_t k = 0; k < own.size(); ++k)
    LB_BTRY(cudaMemcpyAsync(&own[k], b->ctxs[b->runs[k]]->d_status, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
  LB_BTRY(cudaStreamSynchronize(b->stream));
  for (int v : own)
    if (st == 0) st = v;
  return st != 0 ? st : LB_OK;
}

int lb_batch_reduce(lb_batch* b, int32_t want_residual, double* out) {
  if (!b || !out) return LB_E_INVAL;
  DevGuard guard(b->device);
  const size_t n = b->ctxs.size();
  if (!b->d_sums) {
    LB_BTRY(cudaMalloc(reinterpret_cast<void**>(&b->d_sums), n * kReduceFields * sizeof(double)));
    LB_BTRY(cudaMallocHost(reinterpret_cast<void**>(&b->h_sums), n * kReduceFields * sizeof(double)));
  }
  // after the work queued on the members' own streams and the batch's steps
  for (size_t i = 0; i < n; ++i) {
    LB_BTRY(cudaEventRecord(b->ctx_ev[i], b->ctxs[i]->stream));
    LB_BTRY(cudaStreamWaitEvent(b->stream, b->ctx_ev[i], 0));
  }
  for (size_t i = 0; i < n; ++i)
    LB_BTRY(aux_reduce_enqueue(b->ctxs[i], b->stream, b->d_sums + i * kReduceFields, want_residual != 0));
  LB_BTRY(cudaMemcpyAsync(b->h_sums, b->d_sums, n * kReduceFields * sizeof(double), cudaMemcpyDeviceToHost,
                          b->stream));
  // the members' reduction buffers and residual snapshots were used on the
  // batch stream: later work on a member's stream comes after
  LB_BTRY(cudaEventRecord(b->done, b->stream));
  for (lb_ctx* x : b->ctxs) LB_BTRY(cudaStreamWaitEvent(x->stream, b->done, 0));
  LB_BTRY(cudaStreamSynchronize(b->stream));
  for (size_t i = 0; i < n; ++i) {
    double* o = out + 6 * i;
    double mom[3] = {0, 0, 0}, res = 0.0;
    const int rc = reduce_finish(b->ctxs[i], b->h_sums + i * kReduceFields, want_residual != 0, &o[0], mom,
                                 want_residual ? &res : nullptr);
    o[1] = mom[0];
    o[2] = mom[1];
    o[3] = mom[2];
    o[4] = res;
    o[5] = rc == LB_OK ? 0.0 : double(rc);
  }
  return LB_OK;
}

int lb_batch_info(const lb_batch* b, lb_batch_info_t* info) {
  if (!b || !info) return LB_E_INVAL;
  std::memset(info, 0, sizeof(*info));
  info->n_domains = int32_t(b->ctxs.size());
  info->n_classes = int32_t(b->classes.size());
  info->total_nodes = b->total_nodes;
  info->steps_done = b->steps_done;
  for (const auto& c : b->classes) {
    info->work_items += c.n_items;
    info->launches_per_step += 1;
    info->ctas += c.grid;
  }
  return LB_OK;
}

int lb_batch_alone(const lb_batch* b, int32_t* members, int32_t cap) {
  if (!b || cap < 0) return LB_E_INVAL;
  for (size_t k = 0; members && k < b->runs.size() && k < size_t(cap); ++k) members[k] = b->runs[k];
  return int(b->runs.size());
}

void lb_batch_destroy(lb_batch* b) {
  if (!b) return;
  DevGuard guard(b->device);
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (cudaStream_t st : b->lanes) cudaStreamSynchronize(st);
  if (b->graph) cudaGraphExecDestroy(b->graph);
  if (b->rest_graph) cudaGraphExecDestroy(b->rest_graph);
  for (auto& c : b->classes) free_class(c);
  for (auto& c : b->rest) free_class(c);
  if (b->d_status) cudaFree(b->d_status);
  if (b->done) cudaEventDestroy(b->done);
  if (b->fork) cudaEventDestroy(b->fork);
  for (cudaEvent_t e : b->join)
    if (e) cudaEventDestroy(e);
  for (cudaStream_t st : b->side)
    if (st) cudaStreamDestroy(st);
  for (cudaEvent_t e : b->ctx_ev)
    if (e) cudaEventDestroy(e);
  for (cudaEvent_t e : b->lane_ev) cudaEventDestroy(e);
  for (cudaStream_t st : b->lanes) cudaStreamDestroy(st);
  if (b->d_sums) cudaFree(b->d_sums);
  if (b->h_sums) cudaFreeHost(b->h_sums);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

}  // extern "C"
