// lb_cg.cu -- two-component colour-gradient step (paper section 2.1) in the
// thread-safe form of section 4: a node's post-collision set is known from a
// few moment fields, the phase field gradient is taken in a launch of its own,
// and a node's new populations are pulled from the fields of its upstream
// nodes.
//
// Per node x, from the two colours f_R, f_B:
//   rho_R = sum f_R, rho_B = sum f_B, g = f_R + f_B, and the regularized
//   relaxation coefficients of g (lb_collide.cuh: A, B, C, the order-2
//   Hermite form of Eq. LBexp / Eq. hermite), phi = (rho_R - rho_B) / rho,
//   c_R = rho_R / rho and c_RB = beta rho_R rho_B / rho;
// (gradient launch) grad phi = (1/cs2) sum_a t_a c_a phi(x + c_a), stored as
//   |grad phi| and the unit normal n;
// (pull) for every direction a and upstream node x = y - c_a:
//   g*_a = t_a (A + B.c_a + c_a.C.c_a) + (9/4) sigma omega |grad phi|
//          [t_a (c_a.n)^2 - B_a]                          (perturbation)
//   f_R(y)_a = c_R g*_a + c_RB t_a (c_a.n)/|c_a|,  f_B(y)_a = g*_a - f_R(y)_a
//                                                         (recolouring)
// Each colour is stored shifted by half the rest population, t_a rho0 / 2,
// so that g is stored shifted by t_a rho0 as in the single-component path.
// Periodic box only; D2Q9 and D3Q19; FP64 or FP32 storage and arithmetic.
//
// Between two steps of one lb_cg_step() call the populations exist in
// registers only: the step launch pulls them from one set of fields and writes
// the moment fields of the next set.  A run is
//   enter (populations -> set A), gradient A,
//   n - 1 times: step (A -> B or B -> A), gradient of the new set,
//   leave (set A -> populations),
// two launches a step.  Set A has memory of its own; set B lies in the
// population arrays, which the enter launch has read by then, so a run needs an
// odd n (an even one is preceded by a run of one step).  The arithmetic is that of
// populations written and read back at every step, operation by operation.
//
// Layout of a set: quads, 16-byte groups (FP32) of four values of a node, so
// that a pull is 3 (2D) or 4 (3D) vector loads a direction: the coefficients
// with c_R and c_RB behind them, and |grad phi| with n; and phi on its own,
// which the gradient reads at 8 or 18 neighbours.  FP32 bytes per update: the
// step reads 48 and writes 36 (3D: 64 and 52), the gradient reads 4 and writes
// 16: 104 (136), where three launches over populations and planar fields moved
// 284 (444).  Measured per step on one GB300, three launches against this form:
// D2Q9 FP32 4096^2 1126 -> 488 us, 2048 x 1536 with near-contact forces 328 ->
// 137 us, D3Q19 FP32 192^3 933 -> 427 us (bound by the L1's loads of a pull;
// 767 with boxes of 8 nodes along x), 97 x 61 x 113 98.6 -> 58.3 us; FP64 is bound by its arithmetic (1024^2 624 ->
// 613 us).
//
// Near-contact interactions (section 2.2), when switched on: the gradient
// launch also flags node y if, for some direction a, the node y - h c_a is
// bulk (phi < -1 + eps) and both y and y - 2h c_a are not -- the paper's test
// from the bulk node, written from the flagged node so that every thread
// writes only its own node -- and a flagged node's relaxation coefficients
// are recomputed from its own populations with the body force
// F = A rho_R grad phi / |grad phi| (the forcing of the single-component
// step).  Its populations are those in memory at a run's first step, and are
// pulled once more from the set before at the others (flagged nodes line the
// thin films between droplets: few).  No thread reads this set's coefficients
// in that launch, and the set before is only written by the launch after it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "lb_dispatch.cuh"
#include "lb_ptx.cuh"
#include "lb_widen.cuh"

namespace lbgb {
namespace {

constexpr int kCgThreads = 256;
// values per node of a set: NC coefficients, c_R, c_RB; |grad phi| and n (3); phi
constexpr int kCgFields = 17;  // of D3Q19; D2Q9 uses 13

template <class R>
struct alignas(16) Quad {
  R v[4];
};

// one set of fields; quad j of node i is k[j * n + i]
template <class R>
struct CgSet {
  Quad<R>* k;     // the coefficients in the order of each_coef, c_R, c_RB
  Quad<R>* grad;  // |grad phi|, n
  R* phi;
};

// Extents, and the box of nodes a thread block works on: 2^lx x 2^ly x 2^lz =
// kCgThreads nodes (internal axes; 2D: nx x 1 x ny).
struct CgGeom {
  int nx, ny, nz;
  int64_t n;
  int lx, ly, lz;
  uint32_t ntx, nty, ntz;  // boxes along each axis
};

struct CgNode {
  int x, y, z;
  bool in;
};
__device__ __forceinline__ CgNode cg_node(const CgGeom& g) {
  const uint32_t b = blockIdx.x, r = b / g.ntx;
  CgNode o;
  o.x = int((b - r * g.ntx) << g.lx) + int(threadIdx.x & ((1u << g.lx) - 1));
  const uint32_t bz = r / g.nty;
  o.y = int((r - bz * g.nty) << g.ly) + int((threadIdx.x >> g.lx) & ((1u << g.ly) - 1));
  o.z = int(bz << g.lz) + int(threadIdx.x >> (g.lx + g.ly));
  o.in = o.x < g.nx && o.y < g.ny && o.z < g.nz;
  return o;
}

// node index, for coordinates up to one period outside (a domain that fits the
// memory has fewer than 2^31 nodes: 140 bytes each at the least)
__device__ __forceinline__ uint32_t cg_wrap_index(const CgGeom& g, int x, int y, int z) {
  x = x < 0 ? x + g.nx : (x >= g.nx ? x - g.nx : x);
  y = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
  z = z < 0 ? z + g.nz : (z >= g.nz ? z - g.nz : z);
  return uint32_t(x) + uint32_t(g.nx) * (uint32_t(y) + uint32_t(g.ny) * uint32_t(z));
}

// perturbation weights B_a by |c|^2 shell; sum B = cs2, sum B c c = cs2 I
template <class L>
__host__ __device__ constexpr double cg_B(int a) {
  const int c2 = L::cx(a) * L::cx(a) + L::cy(a) * L::cy(a) + L::cz(a) * L::cz(a);
  if (L::ID == LB_D2Q9) return c2 == 0 ? -4.0 / 27.0 : (c2 == 1 ? 2.0 / 27.0 : 5.0 / 108.0);
  return c2 == 0 ? -2.0 / 9.0 : (c2 == 1 ? 1.0 / 54.0 : 1.0 / 27.0);
}

// relaxation coefficients k of a node and c_R, c_RB <-> quads
template <class L, class R>
__device__ __forceinline__ void cg_store_coef(const CgSet<R>& s, int64_t n, uint32_t i, Coef<R>& k, R cr, R crb) {
  constexpr int NC = n_coef<L>();
  Quad<R> q[(NC + 2) / 4];
  each_coef<L, R>(k, [&](auto I, R& v) { q[decltype(I)::value / 4].v[decltype(I)::value % 4] = v; });
  q[NC / 4].v[NC % 4] = cr;
  q[(NC + 1) / 4].v[(NC + 1) % 4] = crb;
#pragma unroll
  for (int j = 0; j < (NC + 2) / 4; ++j) s.k[j * n + i] = q[j];
}

// moment fields of a node from its populations' sums: g (all directions) and
// the two colours' densities, shifted
template <class L, class R>
__device__ __forceinline__ void cg_store_moments(const CgSet<R>& s, int64_t n, uint32_t i, const R (&gt)[L::Q], R sr,
                                                 R sb, const Phys<R>& ph, R half_rho0, R beta) {
  Mom<R> m;
  moments<L, R, false>(gt, ph, m);
  Coef<R> k;
  coeffs<L, R, false>(m, ph, k);
  const R rr = sr + half_rho0, rb = sb + half_rho0, rho = rr + rb;
  cg_store_coef<L>(s, n, i, k, rr / rho, beta * rr * rb / rho);
  s.phi[i] = (rr - rb) / rho;
}

// constants of the pull
template <class R>
struct CgPull {
  R pert_k, half_rho0;  // (9/4) sigma omega, rho0 / 2
};

// the populations that arrive at node (x, y, z): f(a, f_R, f_B), shifted
template <class L, class R, class F>
__device__ __forceinline__ void cg_pull(const CgGeom& g, const CgSet<R>& s, int x, int y, int z, const CgPull<R>& pc,
                                        F&& f) {
  constexpr int NC = n_coef<L>();
  static_for<0, L::Q>([&](auto A_) {
    constexpr int a = decltype(A_)::value;
    constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
    const uint32_t u = cg_wrap_index(g, x - cx, y - cy, z - cz);  // upstream node
    Quad<R> q[(NC + 2) / 4];
#pragma unroll
    for (int j = 0; j < (NC + 2) / 4; ++j) q[j] = s.k[j * g.n + u];
    const Quad<R> gq = s.grad[u];
    Coef<R> k{};
    each_coef<L, R>(k, [&](auto I, R& v) { v = q[decltype(I)::value / 4].v[decltype(I)::value % 4]; });
    const R cr = q[NC / 4].v[NC % 4], crb = q[(NC + 1) / 4].v[(NC + 1) % 4];
    constexpr R w = R(weight<L>(a));
    const R gpost = post<L, R, a>(k) + w * (R(2) * pc.half_rho0);  // unshifted relaxed total population
    const R gn = gq.v[0];
    R cn = R(0);  // c_a . n
    if constexpr (cx != 0) cn = fma_r(R(cx), gq.v[1], cn);
    if constexpr (cy != 0) cn = fma_r(R(cy), gq.v[2], cn);
    if constexpr (cz != 0) cn = fma_r(R(cz), gq.v[3], cn);
    constexpr R B = R(cg_B<L>(a));
    const R gstar = fma_r(pc.pert_k * gn, fma_r(w * cn, cn, -B), gpost);
    constexpr int c2 = cx * cx + cy * cy + cz * cz;
    constexpr R inv_len = c2 == 0 ? R(0) : (c2 == 1 ? R(1) : (c2 == 2 ? R(0.70710678118654752440) :
                                                                   R(0.57735026918962576451)));
    const R rec = crb * (w * (cn * inv_len));
    const R fred = fma_r(cr, gstar, rec);
    const R fblue = gstar - fred;
    f(A_, fred - w * pc.half_rho0, fblue - w * pc.half_rho0);
  });
}

template <class L, class S, class R>
__global__ void __launch_bounds__(kCgThreads) cg_enter_kernel(const CgGeom g, const S* __restrict__ fr,
                                                              const S* __restrict__ fb, const Phys<R> ph,
                                                              R half_rho0, R beta, const CgSet<R> dst) {
  const CgNode o = cg_node(g);
  if (!o.in) return;
  const uint32_t i = cg_wrap_index(g, o.x, o.y, o.z);
  R gt[L::Q];
  R sr = R(0), sb = R(0);
  static_for<0, L::Q>([&](auto A_) {
    constexpr int a = decltype(A_)::value;
    const R r = load_as<S, R>(fr[a * g.n + i]), b = load_as<S, R>(fb[a * g.n + i]);
    sr = sr + r;
    sb = sb + b;
    gt[a] = r + b;
  });
  cg_store_moments<L>(dst, g.n, i, gt, sr, sb, ph, half_rho0, beta);
}

// One step between sets.  Bound by the L1's vector loads and instruction issue
// (a node pulls 9 or 19 directions of 48 or 64 bytes, DRAM sees each set once).
template <class L, class S, class R>
__global__ void __launch_bounds__(kCgThreads) cg_step_kernel(const CgGeom g, const CgSet<R> src, const Phys<R> ph,
                                                             const CgPull<R> pc, R beta, const CgSet<R> dst) {
  grid_wait();  // launch_step
  grid_release();
  const CgNode o = cg_node(g);
  if (!o.in) return;
  R gt[L::Q];
  R sr = R(0), sb = R(0);
  cg_pull<L>(g, src, o.x, o.y, o.z, pc, [&](auto A_, R fr, R fb) {
    const R r = round_to_storage<S, R>(fr), b = round_to_storage<S, R>(fb);
    sr = sr + r;
    sb = sb + b;
    gt[decltype(A_)::value] = r + b;
  });
  cg_store_moments<L>(dst, g.n, cg_wrap_index(g, o.x, o.y, o.z), gt, sr, sb, ph, pc.half_rho0, beta);
}

template <class L, class S, class R>
__global__ void __launch_bounds__(kCgThreads) cg_leave_kernel(const CgGeom g, const CgSet<R> src, const CgPull<R> pc,
                                                              S* __restrict__ fr, S* __restrict__ fb) {
  const CgNode o = cg_node(g);
  if (!o.in) return;
  const uint32_t i = cg_wrap_index(g, o.x, o.y, o.z);
  cg_pull<L>(g, src, o.x, o.y, o.z, pc, [&](auto A_, R r, R b) {
    constexpr int a = decltype(A_)::value;
    fr[a * g.n + i] = store_as<S, R>(r);
    fb[a * g.n + i] = store_as<S, R>(b);
  });
}

// near-contact parameters of the gradient launch
template <class R>
struct CgNci {
  R amp, bulk;  // A, -1 + eps
  int h;
};

// gradient of set s; prev: the set that s was stepped from (PULL), else its
// populations are in fr, fb
template <class L, class S, class R, bool NCI, bool PULL>
__global__ void __launch_bounds__(kCgThreads) cg_gradient_kernel(const CgGeom g, const CgSet<R> s, const CgSet<R> prev,
                                                                  const S* fr, const S* fb, const Phys<R> ph,
                                                                  const CgPull<R> pc, const CgNci<R> nci) {
  grid_wait();  // launch_step
  grid_release();
  const CgNode o = cg_node(g);
  if (!o.in) return;
  const int x = o.x, y = o.y, z = o.z;
  const uint32_t i = cg_wrap_index(g, x, y, z);
  R gv[3] = {R(0), R(0), R(0)};
  static_for<1, L::Q>([&](auto A_) {
    constexpr int a = decltype(A_)::value;
    const R p = s.phi[cg_wrap_index(g, x + L::cx(a), y + L::cy(a), z + L::cz(a))];
    constexpr R w = R(weight<L>(a));
    if constexpr (L::cx(a) != 0) gv[0] = fma_r(R(L::cx(a)) * w, p, gv[0]);
    if constexpr (L::cy(a) != 0) gv[1] = fma_r(R(L::cy(a)) * w, p, gv[1]);
    if constexpr (L::cz(a) != 0) gv[2] = fma_r(R(L::cz(a)) * w, p, gv[2]);
  });
  R g2 = R(0);
  for (int al = 0; al < 3; ++al) {
    gv[al] = gv[al] * R(3);  // 1 / cs2
    g2 = fma_r(gv[al], gv[al], g2);
  }
  const R gn = sqrt(g2);
  Quad<R> gq;
  gq.v[0] = gn;
  for (int al = 0; al < 3; ++al) gq.v[1 + al] = gn > R(0) ? gv[al] / gn : R(0);
  s.grad[i] = gq;
  if constexpr (NCI) {
    bool flag = false;
    if (s.phi[i] > nci.bulk && gn > R(0)) {
      const int h = nci.h;
      // the far samples only beyond near ones in the bulk (few): half the loads
      R p1[L::Q];
      static_for<1, L::Q>([&](auto A_) {
        constexpr int a = decltype(A_)::value;
        p1[a] = s.phi[cg_wrap_index(g, x - h * L::cx(a), y - h * L::cy(a), z - h * L::cz(a))];
      });
      static_for<1, L::Q>([&](auto A_) {
        constexpr int a = decltype(A_)::value;
        if (p1[a] < nci.bulk)
          flag = flag ||
                 s.phi[cg_wrap_index(g, x - 2 * h * L::cx(a), y - 2 * h * L::cy(a), z - 2 * h * L::cz(a))] > nci.bulk;
      });
    }
    if (flag) {
      R gt[L::Q];
      R sr = R(0);
      if constexpr (PULL) {
        cg_pull<L>(g, prev, x, y, z, pc, [&](auto A_, R r0, R b0) {
          const R r = round_to_storage<S, R>(r0), b = round_to_storage<S, R>(b0);
          sr = sr + r;
          gt[decltype(A_)::value] = r + b;
        });
      } else {
        static_for<0, L::Q>([&](auto A_) {
          constexpr int a = decltype(A_)::value;
          const R r = load_as<S, R>(fr[a * g.n + i]), b = load_as<S, R>(fb[a * g.n + i]);
          sr = sr + r;
          gt[a] = r + b;
        });
      }
      const R rr = sr + pc.half_rho0;  // rho_R
      Phys<R> pf = ph;
      for (int al = 0; al < 3; ++al) {
        pf.F[al] = nci.amp * rr * gq.v[1 + al];
        pf.hF[al] = R(0.5) * pf.F[al];
      }
      Mom<R> m;
      moments<L, R, true>(gt, pf, m);
      Coef<R> k;
      coeffs<L, R, true>(m, pf, k);
      // the last quad keeps its c_R and c_RB
      constexpr int NC = n_coef<L>(), last = NC / 4;
      static_assert(NC % 4 == 2, "c_R and c_RB fill the last quad");
      const Quad<R> q = s.k[last * g.n + i];
      cg_store_coef<L>(s, g.n, i, k, q.v[2], q.v[3]);
    }
  }
}

// f_k = (rho_k / rho) f^eq(rho, u) (FP64), stored shifted by t_a rho0 / 2
template <class L, class S>
__global__ void cg_init_kernel(CgGeom g, const double* __restrict__ rr, const double* __restrict__ rb,
                               const double* __restrict__ u, int d, double rho0, S* __restrict__ fr,
                               S* __restrict__ fb) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < g.n; i += int64_t(gridDim.x) * blockDim.x) {
    double uu[3] = {0, 0, 0};
    if (u) {
      uu[0] = u[i];
      if (d == 2) uu[2] = u[g.n + i];  // user y is internal z in 2D
      else {
        uu[1] = u[g.n + i];
        uu[2] = u[2 * g.n + i];
      }
    }
    const double rho = rr[i] + rb[i], usq = uu[0] * uu[0] + uu[1] * uu[1] + uu[2] * uu[2];
    static_for<0, L::Q>([&](auto A_) {
      constexpr int a = decltype(A_)::value;
      const double cu = L::cx(a) * uu[0] + L::cy(a) * uu[1] + L::cz(a) * uu[2];
      const double w = weight<L>(a);
      const double feq = w * (rho + rho0 * (3.0 * cu + 4.5 * cu * cu - 1.5 * usq));
      // S is float or double here: the conversion rounds to nearest
      fr[a * g.n + i] = static_cast<S>(rr[i] / rho * feq - 0.5 * w * rho0);
      fb[a * g.n + i] = static_cast<S>(rb[i] / rho * feq - 0.5 * w * rho0);
    });
  }
}

template <class L, class S, class R>
__global__ void cg_get_kernel(CgGeom g, const S* fs, ShellSums sums, double* f) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < g.n; i += int64_t(gridDim.x) * blockDim.x)
    widen_populations<L, S, R>(fs + i, g.n, f + i, g.n, sums);
}

template <class L, class S, class R>
__global__ void cg_set_kernel(CgGeom g, const double* __restrict__ f, double rho0, S* __restrict__ fs) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < g.n; i += int64_t(gridDim.x) * blockDim.x)
    static_for<0, L::Q>([&](auto A_) {
      constexpr int a = decltype(A_)::value;
      fs[a * g.n + i] = store_as<S, R>(R(f[a * g.n + i] - 0.5 * weight<L>(a) * rho0));
    });
}

template <class L, class S, class R>
__global__ void cg_fields_kernel(CgGeom g, const S* __restrict__ fr, const S* __restrict__ fb, double rho0,
                                 int d, double* __restrict__ rr, double* __restrict__ rb, double* __restrict__ u) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < g.n; i += int64_t(gridDim.x) * blockDim.x) {
    double sr = 0.0, sb = 0.0, j[3] = {0, 0, 0};
    // (the terms with a zero component leave a finite sum as it is; they are
    // added only where a population is not finite)
    bool finite = true;
    static_for<0, L::Q>([&](auto A_) {
      constexpr int a = decltype(A_)::value;
      constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
      const double r = widen(load_as<S, R>(fr[a * g.n + i])), b = widen(load_as<S, R>(fb[a * g.n + i]));
      finite = finite && isfinite(r) && isfinite(b);
      sr += r;
      sb += b;
      const double t = r + b;
      if constexpr (cx != 0) j[0] += cx > 0 ? t : -t;
      if constexpr (cy != 0) j[1] += cy > 0 ? t : -t;
      if constexpr (cz != 0) j[2] += cz > 0 ? t : -t;
    });
    if (!finite) {
      j[0] = j[1] = j[2] = 0.0;
      static_for<0, L::Q>([&](auto A_) {
        constexpr int a = decltype(A_)::value;
        const double t = double(load_as<S, R>(fr[a * g.n + i])) + double(load_as<S, R>(fb[a * g.n + i]));
        j[0] += L::cx(a) * t;
        j[1] += L::cy(a) * t;
        j[2] += L::cz(a) * t;
      });
    }
    if (rr) rr[i] = sr + 0.5 * rho0;
    if (rb) rb[i] = sb + 0.5 * rho0;
    if (u) {
      // (rho0 = 1: lb_cg_create)
      u[i] = j[0];
      if (d == 2) u[g.n + i] = j[2];
      else {
        u[g.n + i] = j[1];
        u[2 * g.n + i] = j[2];
      }
    }
  }
}

int grid_of(int64_t n) {
  int64_t b = (n + kCgThreads - 1) / kCgThreads;
  return int(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

// The box of a thread block: the power-of-two extents whose boxes cover the
// domain at the least cost.  The L1's loads bound the pull: a warp's 16-byte
// load touches one 128-byte line for every 8 nodes of a row and one more for
// each row (shifted rows straddle lines): 5 lines for rows of 32 nodes, 8 for
// rows of 8.  The ring of neighbours that a box reads comes from the L2 cache
// and counts a tenth.
void plan_boxes(CgGeom& g) {
  double best = 1e300;
  for (int lx = 0; lx <= 8; ++lx)
    for (int ly = 0; lx + ly <= 8; ++ly) {
      const int lz = 8 - lx - ly;
      const double bx = 1 << lx, by = 1 << ly, bz = 1 << lz;
      const double tx = std::ceil(g.nx / bx), ty = std::ceil(g.ny / by), tz = std::ceil(g.nz / bz);
      const double ring = (1 + 2 / bx) * (g.ny > 1 ? 1 + 2 / by : 1) * (1 + 2 / bz) - 1;
      const double row = std::min(bx, 32.0);  // of a warp
      const double lines = 32 / row * (std::max(1.0, row / 8) + 1);
      const double cost = tx * ty * tz * (lines / 5 + ring / 10);
      if (cost < best * (1 - 1e-9)) {
        best = cost;
        g.lx = lx;
        g.ly = ly;
        g.lz = lz;
        g.ntx = uint32_t(tx);
        g.nty = uint32_t(ty);
        g.ntz = uint32_t(tz);
      }
    }
}

int rc_of(cudaError_t e) { return e == cudaSuccess ? LB_OK : (e == cudaErrorMemoryAllocation ? LB_E_NOMEM : LB_E_CUDA); }

template <class F>
bool cg_dispatch(int lattice, int storage, F&& f) {
  if (storage != LB_F64 && storage != LB_F32) return false;
  auto on = [&](auto Lt) {
    if (storage == LB_F64) f(Lt, type_tag<double>{}, type_tag<double>{});
    else f(Lt, type_tag<float>{}, type_tag<float>{});
    return true;
  };
  return lattice == LB_D2Q9 ? on(D2Q9{}) : lattice == LB_D3Q19 ? on(D3Q19{}) : false;
}

}  // namespace
}  // namespace lbgb

struct lb_cg {
  int lattice, q, d, storage;
  int64_t dims[3];
  lbgb::CgGeom g;
  double tau, sigma, beta, rho0;
  cudaStream_t stream;
  bool own_stream;
  int device;
  size_t es, rs;  // storage and arithmetic element sizes
  void* fr;
  void* fb;
  void* fld;
  int64_t steps_done;
  double nci_amp, nci_eps;  // near-contact interactions: off while nci_amp == 0
  int nci_h;
};

using namespace lbgb;

namespace {

struct CgDev {
  int prev = -1;
  explicit CgDev(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (dev >= 0 && dev != prev) cudaSetDevice(dev);
  }
  ~CgDev() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

// stage an FP64 buffer to the device (host input) or use it (device input)
int cg_stage(lb_cg* c, const double* src, size_t count, int on_device, double** out, bool* owned) {
  *out = nullptr;
  *owned = false;
  if (!src) return LB_OK;
  if (on_device) {
    *out = const_cast<double*>(src);
    return LB_OK;
  }
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(out), count * sizeof(double), c->stream);
  if (e != cudaSuccess) return rc_of(e);
  *owned = true;
  return rc_of(cudaMemcpyAsync(*out, src, count * sizeof(double), cudaMemcpyHostToDevice, c->stream));
}

}  // namespace

extern "C" {

int lb_cg_create(int32_t lattice, const int64_t dims[3], double tau, double sigma, double beta, int32_t storage,
                 void* stream, lb_cg** out) {
  if (!out || !dims) return LB_E_INVAL;
  *out = nullptr;
  if (lattice != LB_D2Q9 && lattice != LB_D3Q19) return LB_E_UNSUPPORTED;
  if (storage != LB_F64 && storage != LB_F32) return LB_E_UNSUPPORTED;
  const int d = lattice == LB_D2Q9 ? 2 : 3;
  for (int k = 0; k < 3; ++k)
    if (dims[k] < 1 || dims[k] > (int64_t(1) << 30)) return LB_E_INVAL;
  if (d == 2 && dims[2] != 1) return LB_E_INVAL;
  if (!(tau > 0.5) || !(tau < 1e6) || !(sigma >= 0.0) || !(beta >= 0.0) || !(beta <= 1.0)) return LB_E_INVAL;
  lb_cg* c = new (std::nothrow) lb_cg();
  if (!c) return LB_E_NOMEM;
  c->lattice = lattice;
  c->q = lattice == LB_D2Q9 ? 9 : 19;
  c->d = d;
  c->storage = storage;
  for (int k = 0; k < 3; ++k) c->dims[k] = dims[k];
  c->g.nx = int(dims[0]);
  c->g.ny = d == 2 ? 1 : int(dims[1]);
  c->g.nz = d == 2 ? int(dims[1]) : int(dims[2]);
  c->g.n = dims[0] * dims[1] * dims[2];
  plan_boxes(c->g);
  c->tau = tau;
  c->sigma = sigma;
  c->beta = beta;
  c->rho0 = 1.0;
  c->es = c->rs = storage == LB_F64 ? 8 : 4;
  if (cudaGetDevice(&c->device) != cudaSuccess) {
    delete c;
    return LB_E_CUDA;
  }
  int rc = LB_OK;
  do {
    if (stream) {
      c->stream = static_cast<cudaStream_t>(stream);
    } else {
      if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) { rc = LB_E_CUDA; break; }
      c->own_stream = true;
    }
    const size_t pop = size_t(c->q) * size_t(c->g.n) * c->es;
    if ((rc = rc_of(cudaMalloc(&c->fr, pop))) != LB_OK) break;
    if ((rc = rc_of(cudaMalloc(&c->fb, pop))) != LB_OK) break;
    if ((rc = rc_of(cudaMalloc(&c->fld, size_t(kCgFields) * size_t(c->g.n) * c->rs))) != LB_OK) break;
    // an even mixture at rest: each colour t_a rho0 / 2, i.e. zero shifted values
    if ((rc = rc_of(cudaMemsetAsync(c->fr, 0, pop, c->stream))) != LB_OK) break;
    if ((rc = rc_of(cudaMemsetAsync(c->fb, 0, pop, c->stream))) != LB_OK) break;
    rc = rc_of(cudaStreamSynchronize(c->stream));
  } while (false);
  if (rc != LB_OK) {
    lb_cg_destroy(c);
    return rc;
  }
  *out = c;
  return LB_OK;
}

int lb_cg_init(lb_cg* c, const double* rho_r, const double* rho_b, const double* u, int32_t on_device) {
  if (!c || !rho_r || !rho_b) return LB_E_INVAL;
  CgDev guard(c->device);
  double *dr, *db, *du;
  bool o1, o2, o3;
  const size_t N = size_t(c->g.n);
  int rc = cg_stage(c, rho_r, N, on_device, &dr, &o1);
  if (rc == LB_OK) rc = cg_stage(c, rho_b, N, on_device, &db, &o2);
  else o2 = false, db = nullptr;
  if (rc == LB_OK) rc = cg_stage(c, u, N * c->d, on_device, &du, &o3);
  else o3 = false, du = nullptr;
  if (rc == LB_OK) {
    cg_dispatch(c->lattice, c->storage, [&](auto Lt, auto St, auto) {
      using L = decltype(Lt);
      using S = typename decltype(St)::type;
      cg_init_kernel<L, S><<<grid_of(c->g.n), kCgThreads, 0, c->stream>>>(
          c->g, dr, db, du, c->d, c->rho0, static_cast<S*>(c->fr), static_cast<S*>(c->fb));
    });
    rc = rc_of(cudaGetLastError());
  }
  if (o1) cudaFreeAsync(dr, c->stream);
  if (o2) cudaFreeAsync(db, c->stream);
  if (o3) cudaFreeAsync(du, c->stream);
  const int rc2 = rc_of(cudaStreamSynchronize(c->stream));
  return rc != LB_OK ? rc : rc2;
}

int lb_cg_set_populations(lb_cg* c, const double* fr, const double* fb, int32_t on_device) {
  if (!c || !fr || !fb) return LB_E_INVAL;
  CgDev guard(c->device);
  const size_t cnt = size_t(c->q) * size_t(c->g.n);
  int rc = LB_OK;
  for (int k = 0; k < 2 && rc == LB_OK; ++k) {
    double* d;
    bool owned;
    rc = cg_stage(c, k == 0 ? fr : fb, cnt, on_device, &d, &owned);
    if (rc != LB_OK) break;
    cg_dispatch(c->lattice, c->storage, [&](auto Lt, auto St, auto Rt) {
      using L = decltype(Lt);
      using S = typename decltype(St)::type;
      using R = typename decltype(Rt)::type;
      cg_set_kernel<L, S, R><<<grid_of(c->g.n), kCgThreads, 0, c->stream>>>(c->g, d, c->rho0,
                                                                            static_cast<S*>(k == 0 ? c->fr : c->fb));
    });
    rc = rc_of(cudaGetLastError());
    if (owned) cudaFreeAsync(d, c->stream);
  }
  const int rc2 = rc_of(cudaStreamSynchronize(c->stream));
  return rc != LB_OK ? rc : rc2;
}

int lb_cg_get_populations(lb_cg* c, double* fr, double* fb, int32_t on_device) {
  if (!c || (!fr && !fb)) return LB_E_INVAL;
  CgDev guard(c->device);
  const size_t cnt = size_t(c->q) * size_t(c->g.n);
  int rc = LB_OK;
  for (int k = 0; k < 2 && rc == LB_OK; ++k) {
    double* dst = k == 0 ? fr : fb;
    if (!dst) continue;
    double* d = dst;
    if (!on_device) {
      rc = rc_of(cudaMallocAsync(reinterpret_cast<void**>(&d), cnt * sizeof(double), c->stream));
      if (rc != LB_OK) break;
    }
    cg_dispatch(c->lattice, c->storage, [&](auto Lt, auto St, auto Rt) {
      using L = decltype(Lt);
      using S = typename decltype(St)::type;
      using R = typename decltype(Rt)::type;
      cg_get_kernel<L, S, R><<<grid_of(c->g.n), kCgThreads, 0, c->stream>>>(
          c->g, static_cast<const S*>(k == 0 ? c->fr : c->fb), shell_sums<L>(0.5 * c->rho0), d);
    });
    rc = rc_of(cudaGetLastError());
    if (!on_device) {
      if (rc == LB_OK) rc = rc_of(cudaMemcpyAsync(dst, d, cnt * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
      cudaFreeAsync(d, c->stream);
    }
  }
  const int rc2 = rc_of(cudaStreamSynchronize(c->stream));
  return rc != LB_OK ? rc : rc2;
}

int lb_cg_step(lb_cg* c, int64_t n) {
  if (!c || n < 0) return LB_E_INVAL;
  CgDev guard(c->device);
  Geometry geo{};
  geo.tau = c->tau;
  geo.rho0 = c->rho0;
  // runs of an odd number of steps end in set A; an even n takes one step first
  while (n > 0) {
    const int64_t run = n % 2 ? n : 1;
    cg_dispatch(c->lattice, c->storage, [&](auto Lt, auto St, auto Rt) {
      using L = decltype(Lt);
      using S = typename decltype(St)::type;
      using R = typename decltype(Rt)::type;
      const Phys<R> ph = make_phys<R>(geo);
      const CgPull<R> pc{R(2.25 * c->sigma / c->tau), R(0.5 * c->rho0)};
      const CgNci<R> nci{R(c->nci_amp), R(-1.0 + c->nci_eps), c->nci_h};
      S* fr = static_cast<S*>(c->fr);
      S* fb = static_cast<S*>(c->fb);
      // set A in fld; set B: the coefficients in f_R's array, the rest in f_B's
      // (NC + 2 <= q and 4 + 1 <= q values a node)
      static_assert(n_coef<L>() + 2 <= L::Q && 5 <= L::Q, "set B fits the population arrays");
      R* fld = static_cast<R*>(c->fld);
      const int64_t N = c->g.n;
      constexpr int NK = n_coef<L>() + 2;
      auto quads = [](R* p) { return reinterpret_cast<Quad<R>*>(p); };
      const CgSet<R> set[2] = {{quads(fld), quads(fld + NK * N), fld + (NK + 4) * N},
                               {quads(reinterpret_cast<R*>(fr)), quads(reinterpret_cast<R*>(fb)),
                                reinterpret_cast<R*>(fb) + 4 * N}};
      const int grid = int(c->g.ntx * c->g.nty * c->g.ntz);
      // about one wave of the step's blocks (128 x 96 D2Q9 FP32: 10.7 -> 5.7 us a step)
      const bool early = grid <= 4 * k1_sm_count();
      auto gradient = [&](int which, auto pull) {
        constexpr bool P = decltype(pull)::value;
        launch_step(c->nci_amp != 0.0 ? cg_gradient_kernel<L, S, R, true, P> : cg_gradient_kernel<L, S, R, false, false>,
                    grid, kCgThreads, 0, c->stream, early, c->g, set[which], set[1 - which],
                    static_cast<const S*>(fr), static_cast<const S*>(fb), ph, pc, nci);
      };
      cg_enter_kernel<L, S, R>
          <<<grid, kCgThreads, 0, c->stream>>>(c->g, fr, fb, ph, pc.half_rho0, R(c->beta), set[0]);
      gradient(0, std::false_type{});
      for (int64_t k = 1; k < run; ++k) {
        const int src = int(k - 1) & 1;
        launch_step(cg_step_kernel<L, S, R>, grid, kCgThreads, 0, c->stream, early, c->g, set[src], ph, pc, R(c->beta),
                    set[1 - src]);
        gradient(1 - src, std::true_type{});
      }
      cg_leave_kernel<L, S, R><<<grid, kCgThreads, 0, c->stream>>>(c->g, set[0], pc, fr, fb);
    });
    if (cudaGetLastError() != cudaSuccess) return LB_E_CUDA;
    c->steps_done += run;
    n -= run;
  }
  return LB_OK;
}

int lb_cg_fields(lb_cg* c, double* rho_r, double* rho_b, double* u, int32_t on_device) {
  if (!c || (!rho_r && !rho_b && !u)) return LB_E_INVAL;
  CgDev guard(c->device);
  const size_t N = size_t(c->g.n);
  double* tmp = nullptr;
  double *dr = rho_r, *db = rho_b, *du = u;
  if (!on_device) {
    int rc = rc_of(cudaMallocAsync(reinterpret_cast<void**>(&tmp), (2 + c->d) * N * sizeof(double), c->stream));
    if (rc != LB_OK) return rc;
    dr = rho_r ? tmp : nullptr;
    db = rho_b ? tmp + N : nullptr;
    du = u ? tmp + 2 * N : nullptr;
  }
  cg_dispatch(c->lattice, c->storage, [&](auto Lt, auto St, auto Rt) {
    using L = decltype(Lt);
    using S = typename decltype(St)::type;
    using R = typename decltype(Rt)::type;
    cg_fields_kernel<L, S, R><<<grid_of(c->g.n), kCgThreads, 0, c->stream>>>(
        c->g, static_cast<const S*>(c->fr), static_cast<const S*>(c->fb), c->rho0, c->d, dr, db, du);
  });
  int rc = rc_of(cudaGetLastError());
  if (!on_device) {
    if (rc == LB_OK && rho_r) rc = rc_of(cudaMemcpyAsync(rho_r, dr, N * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    if (rc == LB_OK && rho_b) rc = rc_of(cudaMemcpyAsync(rho_b, db, N * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    if (rc == LB_OK && u)
      rc = rc_of(cudaMemcpyAsync(u, du, c->d * N * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    cudaFreeAsync(tmp, c->stream);
  }
  const int rc2 = rc_of(cudaStreamSynchronize(c->stream));
  return rc != LB_OK ? rc : rc2;
}

int lb_cg_set_nci(lb_cg* c, double amplitude, double eps, int32_t h) {
  if (!c || !std::isfinite(amplitude) || amplitude < 0.0 || !(eps > 0.0) || !(eps < 2.0) || h < 1) return LB_E_INVAL;
  // the sampled points lie up to 2h nodes away along every moving axis: one
  // periodic wrap must reach them
  const int lim = c->d == 2 ? std::min(c->g.nx, c->g.nz) : std::min(c->g.nx, std::min(c->g.ny, c->g.nz));
  if (2 * int64_t(h) > lim) return LB_E_INVAL;
  c->nci_amp = amplitude;
  c->nci_eps = eps;
  c->nci_h = h;
  return LB_OK;
}

int lb_cg_sync(lb_cg* c) {
  if (!c) return LB_E_INVAL;
  CgDev guard(c->device);
  return rc_of(cudaStreamSynchronize(c->stream));
}

void lb_cg_destroy(lb_cg* c) {
  if (!c) return;
  CgDev guard(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  if (c->fr) cudaFree(c->fr);
  if (c->fb) cudaFree(c->fb);
  if (c->fld) cudaFree(c->fld);
  if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
  delete c;
}

}  // extern "C"
