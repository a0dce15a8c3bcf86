// lb_k3_plan.cu -- runs of several steps in moment form: which contexts take
// them, their sweep length and TMA descriptors, and the sequence of launches.
#include <algorithm>

#include "lb_k3_launch.cuh"

namespace lbgb {

extern const K3Variant k3_variants_d3q19[];
extern const int k3_n_variants_d3q19;
extern const K3Variant k3_variants_d3q27[];
extern const int k3_n_variants_d3q27;
extern const LeaveVariant leave_variants_d3q19[];
extern const int leave_n_variants_d3q19;
extern const LeaveVariant leave_variants_d3q27[];
extern const int leave_n_variants_d3q27;

namespace {

// The first compiled tile of the storage type; domains of up to
// kSmallDomainNodes take the last one, whose more and smaller bricks (two to an
// SM) shorten the sweep that such a step waits for.  Measured, us per step of
// D3Q19 FP32 cavities, 32 x 16 against 32 x 4 tiles: 24^3 5.1 / 4.1, 32^3
// 5.4 / 4.3, 64^3 9.0 / 10.0, 97 x 61 x 113 21.6 / 28.2.
constexpr int64_t kSmallDomainNodes = 65536;

const K3Variant* find_k3(const Geometry& g, int storage) {
  const K3Variant* v =
      g.lattice == LB_D3Q19 ? k3_variants_d3q19 : g.lattice == LB_D3Q27 ? k3_variants_d3q27 : nullptr;
  const int n = g.lattice == LB_D3Q19 ? k3_n_variants_d3q19 : g.lattice == LB_D3Q27 ? k3_n_variants_d3q27 : 0;
  const bool small = int64_t(g.nx) * g.ny * g.nz <= kSmallDomainNodes;
  const K3Variant* found = nullptr;
  for (int i = 0; i < n; ++i)
    if (v[i].storage == storage && (!found || small)) found = &v[i];
  return found;
}

const LeaveVariant* find_leave(int lattice, int storage, int bx, int by) {
  const LeaveVariant* v =
      lattice == LB_D3Q19 ? leave_variants_d3q19 : lattice == LB_D3Q27 ? leave_variants_d3q27 : nullptr;
  const int n = lattice == LB_D3Q19 ? leave_n_variants_d3q19 : lattice == LB_D3Q27 ? leave_n_variants_d3q27 : 0;
  for (int i = 0; i < n; ++i)
    if (v[i].storage == storage && v[i].bx == bx && v[i].by == by) return &v[i];
  return nullptr;
}

// Sweep length: the bricks run in waves of `slots` resident CTAs, and a brick
// costs its planes, the two outer planes and the latency of its first loads
// (about three planes' time).
int choose_bz(int nz, int64_t columns, int slots) {
  int best_bz = nz;
  double best = 1e300;
  for (int n = 1; n <= nz; ++n) {
    const int bz = (nz + n - 1) / n;
    const int64_t bricks = columns * ((nz + bz - 1) / bz);
    const double cost = double((bricks + slots - 1) / slots) * (bz + 5);
    if (cost < best - 1e-9) {
      best = cost;
      best_bz = bz;
    }
  }
  return best_bz;
}

}  // namespace

size_t moment_scratch_elems(const Geometry& g, int storage) {
  const K3Variant* v = find_k3(g, storage);
  if (!v) return 0;
  return size_t(moment_edge_at(g, storage)) + 2 * size_t(moment_edge_elems(g, v->bx));
}

bool moment_plan(lb_ctx* ctx) {
  MomentRun& m = ctx->mr;
  if (m.state != 0) return m.state > 0;
  m.state = -1;
  if (ctx->scheme != LB_SCHEME_FUSED || ctx->g.zlink[0] || ctx->g.zlink[1]) return false;
  m.v = find_k3(ctx->g, ctx->storage);
  m.lv = find_leave(ctx->lattice, ctx->storage, ctx->plan.bx, ctx->plan.by);
  if (!m.v || (!m.lv && !m.v->leave)) return false;
  if (ctx->f_alloc < moment_scratch_elems(ctx->g, ctx->storage) * ctx->real_bytes) return false;
  const Geometry& g = ctx->g;
  m.bz = choose_bz(g.nz, int64_t(div_up(g.nx, m.v->bx)) * div_up(g.ny, m.v->by), k1_sm_count() * m.v->minb);
  const int nc = g.d == 2 ? 6 : 10;
  bool ok = !m.lv || make_field_map(ctx, &m.tmap_leave, ctx->f, nc, m.lv->bx, m.lv->by);
  for (int set = 0; set < 2; ++set) {
    void* base = static_cast<char*>(ctx->f) + size_t(moment_set_at(g, ctx->storage, set)) * ctx->real_bytes;
    ok = ok && make_field_map(ctx, &m.maps[set], base, nc, m.v->bx, m.v->by);
  }
  if (!ok) return false;
  if (m.v->configure() != cudaSuccess || (m.lv && m.lv->configure() != cudaSuccess)) {
    cudaGetLastError();
    return false;
  }
  m.state = 1;
  return true;
}

namespace {

// kMomentGraphSteps steps A -> B -> ... -> A recorded once as a CUDA graph;
// false (no error left set) where the stream cannot be captured
bool capture_steps(lb_ctx* ctx) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone ||
      cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < kMomentGraphSteps && e == cudaSuccess; ++i) e = ctx->mr.v->step(ctx, i & 1);
  cudaGraph_t graph = nullptr;
  const cudaError_t ee = cudaStreamEndCapture(ctx->stream, &graph);
  cudaGraphExec_t exec = nullptr;
  if (e == cudaSuccess && ee == cudaSuccess && graph) e = cudaGraphInstantiate(&exec, graph, 0);
  else e = cudaErrorStreamCaptureInvalidated;
  if (graph) cudaGraphDestroy(graph);
  cudaGetLastError();
  if (e != cudaSuccess || !exec) return false;
  ctx->mr.graph = exec;
  return true;
}

}  // namespace

cudaError_t moment_run(lb_ctx* ctx, int64_t n) {
  MomentRun& m = ctx->mr;
  // the last step leaves from set A: an odd number of launches starts from B,
  // or, where the populations lie in set B's place, after a single step
  cudaError_t e = cudaSuccess;
  if (m.v->leave && n % 2 == 0) {
    e = k1_step(ctx);
    // the run ends by rebuilding the shell that this step read, so that launches
    // recorded by a caller can be replayed: each time they find their shell
    if (e == cudaSuccess) ctx->parity = 1 - ctx->parity;
    --n;
  }
  const int64_t launches = n - 1;
  int src = int(launches & 1);
  if (e == cudaSuccess) e = m.v->enter(ctx, src);
  int64_t i = 0;
  if (e == cudaSuccess && src) {
    e = m.v->step(ctx, 1);
    ++i;
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool replay = launches - i >= kMomentGraphSteps && cudaStreamIsCapturing(ctx->stream, &cs) == cudaSuccess &&
                      cs == cudaStreamCaptureStatusNone;
  if (replay && e == cudaSuccess && (m.graph || capture_steps(ctx)))
    for (; i + kMomentGraphSteps <= launches && e == cudaSuccess; i += kMomentGraphSteps)
      e = cudaGraphLaunch(m.graph, ctx->stream);
  for (src = 0; i < launches && e == cudaSuccess; ++i, src = 1 - src) e = m.v->step(ctx, src);
  if (m.v->leave) {
    if (e == cudaSuccess) e = m.v->leave(ctx);
    return e == cudaSuccess ? k1_bootstrap(ctx) : e;
  }
  if (e == cudaSuccess) e = m.lv->shell(ctx);
  return e == cudaSuccess ? m.lv->leave(ctx) : e;
}

cudaError_t moment_run_beside(lb_ctx* ctx, int64_t n) {
  if (!moment_plan(ctx)) return cudaErrorInvalidValue;
  if (ctx->beside.state != 1) {
    ctx->beside = ctx->mr;
    ctx->beside.graph = nullptr;
    ctx->beside.shared = true;
  }
  std::swap(ctx->mr, ctx->beside);
  const cudaError_t e = moment_run(ctx, n);
  std::swap(ctx->mr, ctx->beside);
  return e;
}

void drop_moment_run(lb_ctx* ctx) {
  for (MomentRun* m : {&ctx->mr, &ctx->beside}) {
    if (m->graph) cudaGraphExecDestroy(m->graph);
    *m = MomentRun{};
  }
}

}  // namespace lbgb
