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

const K3Variant* find_k3(int lattice, int storage) {
  const K3Variant* v = lattice == LB_D3Q19 ? k3_variants_d3q19 : lattice == LB_D3Q27 ? k3_variants_d3q27 : nullptr;
  const int n = lattice == LB_D3Q19 ? k3_n_variants_d3q19 : lattice == LB_D3Q27 ? k3_n_variants_d3q27 : 0;
  for (int i = 0; i < n; ++i)
    if (v[i].storage == storage) return &v[i];
  return nullptr;
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
  if (!find_k3(g.lattice, storage)) return 0;
  return size_t(g.d == 2 ? 12 : 20) * size_t(g.vol);
}

bool moment_plan(lb_ctx* ctx) {
  MomentRun& m = ctx->mr;
  if (m.state != 0) return m.state > 0;
  m.state = -1;
  if (ctx->scheme != LB_SCHEME_FUSED || ctx->g.zlink[0] || ctx->g.zlink[1]) return false;
  m.v = find_k3(ctx->lattice, ctx->storage);
  m.lv = find_leave(ctx->lattice, ctx->storage, ctx->plan.bx, ctx->plan.by);
  if (!m.v || !m.lv) return false;
  if (ctx->f_alloc < moment_scratch_elems(ctx->g, ctx->storage) * ctx->real_bytes) return false;
  const Geometry& g = ctx->g;
  m.bz = choose_bz(g.nz, int64_t(div_up(g.nx, m.v->bx)) * div_up(g.ny, m.v->by), k1_sm_count() * m.v->minb);
  const int nc = g.d == 2 ? 6 : 10;
  char* f = static_cast<char*>(ctx->f);
  if (!make_field_map(ctx, &m.tmap_a, f, nc, m.v->bx, m.v->by) ||
      !make_field_map(ctx, &m.tmap_b, f + size_t(nc) * size_t(g.vol) * ctx->real_bytes, nc, m.v->bx, m.v->by) ||
      !make_field_map(ctx, &m.tmap_leave, f, nc, m.lv->bx, m.lv->by))
    return false;
  if (m.v->configure() != cudaSuccess || m.lv->configure() != cudaSuccess) {
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
  // the last step leaves from set A: an odd number of launches starts from B
  const int64_t launches = n - 1;
  int src = int(launches & 1);
  cudaError_t e = m.v->enter(ctx, src);
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
  if (e == cudaSuccess) e = m.lv->shell(ctx);
  if (e == cudaSuccess) e = m.lv->leave(ctx);
  if (e == cudaSuccess) ctx->parity = 1 - ctx->parity;
  return e;
}

void drop_moment_run(lb_ctx* ctx) {
  if (ctx->mr.graph) cudaGraphExecDestroy(ctx->mr.graph);
  ctx->mr = MomentRun{};
}

}  // namespace lbgb
