// lb_k3_launch.cuh -- host-side launchers of the step in moment form, one set
// per compiled tile shape, and of the brick launches that end a run.
#pragma once

#include <algorithm>

#include "lb_k1_launch.cuh"
#include "lb_k3.cuh"

namespace lbgb {

// A compiled tile of k3_step (lattice x storage x bx x by).
struct K3Variant {
  int lattice, storage, bx, by, ns, minb;
  cudaError_t (*configure)();
  // one step of the context's domain: set src (0 = A, 1 = B) to the other
  cudaError_t (*step)(lb_ctx*, int src);
  cudaError_t (*enter)(lb_ctx*, int dst);  // populations -> coefficient set dst
  // 16-bit storage: the last step, set A -> populations (else null, see LeaveVariant)
  cudaError_t (*leave)(lb_ctx*);
};

// The launches that end a run for contexts whose brick cross-section is
// bx x by: the shell from coefficient set A, and the last step from set A to
// the populations.  The last step reads the shell that is not current and
// writes the current one, so that a run of any length leaves the parity as it
// was (recorded launches can be replayed, and a batch uploads no parities).
struct LeaveVariant {
  int lattice, storage, bx, by;
  cudaError_t (*configure)();
  cudaError_t (*shell)(lb_ctx*);
  cudaError_t (*leave)(lb_ctx*);
};

template <class L, class S, class R, int BX, int BY, int NS, int MINB>
struct K3Impl {
  using Sh = K3Shape<L, R, BX, BY, NS, MINB>;
  static constexpr bool HALF = sizeof(S) == 2;

  static cudaError_t configure() {
    cudaError_t e = cudaFuncSetAttribute(k3_step<L, S, R, BX, BY, NS, false, MINB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, int(Sh::SMEM));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k3_step<L, S, R, BX, BY, NS, true, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(Sh::SMEM));
    if constexpr (HALF)
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k3_step<L, S, R, BX, BY, NS, false, MINB, true>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(Sh::SMEM));
    return e;
  }

  static R* coef_set(lb_ctx* ctx, int which) {
    return static_cast<R*>(ctx->f) + moment_set_at(ctx->g, ctx->storage, which);
  }

  // the edge records of a set, after the two sets (moment_scratch_elems)
  static R* edges(lb_ctx* ctx, int which) {
    return static_cast<R*>(ctx->f) + moment_edge_at(ctx->g, ctx->storage) + which * moment_edge_elems(ctx->g, BX);
  }

  static K3Args<R> args_of(lb_ctx* ctx, int src) {
    const Geometry& g = ctx->g;
    K3Args<R> a;
    a.ph = make_phys<R>(g);
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.pitch = g.pitch;
    a.vol = g.vol;
    a.vol32 = uint32_t(g.vol / 32);
    for (int k = 0; k < 3; ++k) a.per[k] = g.per[k];
    a.bz = ctx->mr.bz;
    a.ntx = div_up(g.nx, BX);
    a.nty = div_up(g.ny, BY);
    a.ntz = div_up(g.nz, a.bz);
    a.src = coef_set(ctx, src);
    a.dst = coef_set(ctx, 1 - src);
    a.esrc = edges(ctx, src);
    a.edst = edges(ctx, 1 - src);
    a.status = ctx->d_status;
    for (int i = 0; i < 27; ++i)
      for (int j = 0; j < 8; ++j) a.bb[i][j] = R(0);
    a.pop = ctx->f;
    make_bounce_terms<L, R>(g, a.bb);
    return a;
  }

  static cudaError_t step(lb_ctx* ctx, int src) {
    const K3Args<R> a = args_of(ctx, src);
    const int grid = a.ntx * a.nty * a.ntz;
    const CUtensorMap& tm = ctx->mr.maps[src];
    const bool early = !ctx->mr.shared && grid <= k1_sm_count() * MINB;
    return launch_step(ctx->g.has_force ? k3_step<L, S, R, BX, BY, NS, true, MINB>
                                        : k3_step<L, S, R, BX, BY, NS, false, MINB>,
                       grid, Sh::NT, Sh::SMEM, ctx->stream, early, tm, a);
  }

  // (no collision: one instantiation serves with and without a force)
  static cudaError_t leave(lb_ctx* ctx) {
    if constexpr (HALF) {
      const K3Args<R> a = args_of(ctx, 0);
      k3_step<L, S, R, BX, BY, NS, false, MINB, true>
          <<<a.ntx * a.nty * a.ntz, Sh::NT, Sh::SMEM, ctx->stream>>>(ctx->mr.maps[0], a);
    }
    return cudaGetLastError();
  }

  static cudaError_t enter(lb_ctx* ctx, int dst) {
    const Geometry& g = ctx->g;
    const int64_t blocks = std::min<int64_t>((g.vol + 255) / 256, int64_t(1) << 30);
    const S* f = static_cast<const S*>(ctx->f);
    const int64_t rows = int64_t(g.ny) * g.nz;
    if (g.has_force)
      k3_enter<L, S, R, true><<<int(blocks), 256, 0, ctx->stream>>>(f, coef_set(ctx, dst), edges(ctx, dst), g.vol, g.nx,
                                                                    rows, int(g.pitch), BX, make_phys<R>(g));
    else
      k3_enter<L, S, R, false><<<int(blocks), 256, 0, ctx->stream>>>(f, coef_set(ctx, dst), edges(ctx, dst), g.vol,
                                                                     g.nx, rows, int(g.pitch), BX, make_phys<R>(g));
    return cudaGetLastError();
  }

  static constexpr K3Variant variant(int lattice, int storage) {
    return K3Variant{lattice, storage, BX, BY, NS, MINB, &configure, &step, &enter, HALF ? &leave : nullptr};
  }
};

template <class L, class S, class R, int BX, int BY, int NS>
struct LeaveImpl {
  using Sh = K1Shape<L, S, R, BX, BY, NS, 2, 0>;

  static cudaError_t configure() {
    cudaError_t e = cudaFuncSetAttribute(k1_leave_step<L, S, R, BX, BY, NS, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, int(Sh::SMEM));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k1_leave_step<L, S, R, BX, BY, NS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(Sh::SMEM));
    return e;
  }

  static cudaError_t shell(lb_ctx* ctx) {
    K1Args<R> a = k1_make_args<R>(ctx, ctx->parity, 1 - ctx->parity);
    // the coefficients already hold the forcing: one instantiation serves both
    k1_bootstrap<L, S, R, BX, BY, false, true><<<k1_bootstrap_blocks(ctx->g, BX), 256, 0, ctx->stream>>>(a);
    return cudaGetLastError();
  }

  static cudaError_t leave(lb_ctx* ctx) {
    K1Args<R> a = k1_make_args<R>(ctx, 1 - ctx->parity, ctx->parity);
    make_bounce_terms<L, R>(ctx->g, a.bb);
    const int grid = ctx->plan.nbx * ctx->plan.nby * ctx->plan.nbz;
    if (ctx->g.has_force)
      k1_leave_step<L, S, R, BX, BY, NS, true><<<grid, Sh::NT, Sh::SMEM, ctx->stream>>>(ctx->mr.tmap_leave, a);
    else
      k1_leave_step<L, S, R, BX, BY, NS, false><<<grid, Sh::NT, Sh::SMEM, ctx->stream>>>(ctx->mr.tmap_leave, a);
    return cudaGetLastError();
  }

  static constexpr LeaveVariant variant(int lattice, int storage) {
    return LeaveVariant{lattice, storage, BX, BY, &configure, &shell, &leave};
  }
};

}  // namespace lbgb
