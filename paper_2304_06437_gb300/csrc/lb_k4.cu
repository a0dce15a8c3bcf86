// lb_k4.cu -- runs of several steps of 2D domains, several steps per launch.
//
// A 2D tile with a ring of T nodes around it fits shared memory, so one launch
// reads a tile, takes T steps on it and writes it: 2 n_coef values an update
// shrink to (2 + ring) n_coef / T, and a domain of a few tiles takes T steps
// for one launch and one memory latency.  What is left bounds the step:
// instruction issue (large domains) and the launch (small ones).  Per step on
// one GB300, single-step launches against this form: FP32 cavities of 4096^2 328
// -> 97 us (173 GLUPS), 1024^2 43.8 -> 8.2, 301 x 257 18.6 -> 1.5, 128 x 96 14.5 ->
// 1.2; FP64 1024^2 219 -> 173 (bound by the FP64 rate), 301 x 257 72.9 -> 26.0.
//
// Between launches the state of a node is its post-collision coefficients, as
// in lb_k3.cuh (6 values).  The first launch of a run reads populations and the
// last one writes them; set A of the coefficients lies behind the populations
// and set B in their place, so a run is an even number of launches,
//   populations -> A (-> B -> A ...) -> populations,
// with the n steps spread evenly over them, and the shells are rebuilt at its
// end.  Arithmetic and rounding are those of single steps, so the populations
// are bit for bit the same.
//
// In shared memory the tile holds the post-collision populations, each in one
// place (the AA pattern): slot (a, x) holds f*_a of node x before an odd step.
// An odd step of node x takes direction a from slot (a, x - c_a) and leaves its
// own f*_opp(a) there; an even step then finds direction a in slot (opp(a), x)
// and leaves f*_a in slot (a, x).  Every slot belongs to one node in a step: one
// buffer and one barrier a step.  A link through a wall comes from slot
// (opp(a), x) in both (no node but x touches it).  The region that is still
// exact shrinks by one node a step on the sides without a wall, and after T
// steps is the tile.
#include <algorithm>
#include <cmath>

#include "lb_k1_launch.cuh"

namespace lbgb {
namespace {

constexpr int kWidth = 64;   // columns of a tile and its ring
constexpr int kMaxSteps = 8; // steps of one launch
constexpr size_t kTileSmem = size_t(113) * 1024;  // two CTAs to an SM

template <class R>
constexpr int k4_threads() { return sizeof(R) == 8 ? 256 : 512; }
template <class R>
constexpr int k4_max_rows() { return int(kTileSmem / (9 * kWidth * sizeof(R))); }

template <class R>
struct K4Args {
  Phys<R> ph;
  int nx, nz;             // internal extents
  int64_t pitch, vol;
  int per_x, per_z;
  int steps, bx, bz, ntx; // of this launch: steps (the ring's width), tile, tiles along x
  const R* src;           // coefficient set or populations read, and
  R* dst;                 // written: field i at + i * vol
  R bb[27][8];
};

// FROM: the source is populations; TO: so is the destination
template <class R, bool FORCE, bool FROM, bool TO>
__global__ void __launch_bounds__(k4_threads<R>(), 2) k4_steps(const __grid_constant__ K4Args<R> args) {
  using L = D2Q9;
  constexpr int Q = L::Q, NC = n_coef<L>();
  constexpr int ROWS = k4_threads<R>() / kWidth;  // rows per pass
  constexpr int RS = Q * kWidth;                  // slots per row: [direction][column]
  extern __shared__ __align__(128) unsigned char smem[];
  R* const S = reinterpret_cast<R*>(smem);

  const int T = args.steps, nx = args.nx, nz = args.nz;
  const int tI = int(blockIdx.x) % args.ntx, tK = int(blockIdx.x) / args.ntx;
  const int x0 = tI * args.bx, z0 = tK * args.bz;
  const int bxa = min(args.bx, nx - x0), bza = min(args.bz, nz - z0);
  const int tx = threadIdx.x % kWidth, ty = threadIdx.x / kWidth;
  const int gx = x0 - T + tx;  // this thread's column in the domain (unwrapped)

  // columns and rows [lo, hi) that are exact after t steps: t from the edge of
  // what was read, or up to the walls
  auto lo_of = [&](int t, int at, bool per) { return per ? t : max(t, T - at); };
  auto hi_of = [&](int t, int at, int b, int n, bool per) {
    return per ? 2 * T + b - t : min(2 * T + b - t, T + n - at);
  };
  auto wrap = [](int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
  };

  // what came before may still run up to here (launch_step)
  grid_wait();
  grid_release();
  {  // read the tile and its ring
    const bool in = tx >= lo_of(0, x0, args.per_x) && tx < hi_of(0, x0, bxa, nx, args.per_x);
    const int rhi = hi_of(0, z0, bza, nz, args.per_z);
    const R* const col = args.src + wrap(gx, nx);
    for (int r = lo_of(0, z0, args.per_z) + ty; r < rhi; r += ROWS) {
      if (!in) continue;
      const R* p = col + args.pitch * wrap(z0 - T + r, nz);
      Coef<R> k{};
      if constexpr (FROM) {
        R f[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) f[a] = p[a * args.vol];
        moments_coeffs<L, FORCE>(f, args.ph, k);
      } else {
        each_coef<L, R>(k, [&](auto I, R& v) { v = p[decltype(I)::value * args.vol]; });
      }
      R out[Q];
      post_all<L, R>(k, out);
#pragma unroll
      for (int a = 0; a < Q; ++a) S[r * RS + a * kWidth + tx] = out[a];
    }
  }

  // links of this thread's column through an x wall: bit 0 low side, bit 1 high
  const int xw = args.per_x ? 0 : (gx == 0 ? 1 : 0) | (gx == nx - 1 ? 2 : 0);

  auto step = [&](const int t, auto odd_tag, auto wall_tag) {
    constexpr bool ODD = decltype(odd_tag)::value, WALL = decltype(wall_tag)::value;
    const bool last = t == T;
    const bool in = tx >= lo_of(t, x0, args.per_x) && tx < hi_of(t, x0, bxa, nx, args.per_x);
    const int rhi = hi_of(t, z0, bza, nz, args.per_z);
    if (!in) return;
    for (int r = lo_of(t, z0, args.per_z) + ty; r < rhi; r += ROWS) {
      R* const s = S + r * RS + tx;
      const int gz = z0 - T + r;
      int zw = 0;
      if constexpr (WALL) zw = args.per_z ? 0 : (gz == 0 ? 1 : 0) | (gz == nz - 1 ? 2 : 0);
      // bits of the faces through which the link of direction a leaves
      auto combo = [&](auto A_) {
        constexpr int a = decltype(A_)::value;
        int c = 0;
        if constexpr (WALL && L::cx(a) == 1) c |= xw & 1;
        if constexpr (WALL && L::cx(a) == -1) c |= xw >> 1;
        if constexpr (WALL && L::cz(a) == 1) c |= (zw & 1) << 2;
        if constexpr (WALL && L::cz(a) == -1) c |= (zw & 2) << 1;
        return c;
      };
      // the slot that direction a is taken from in an odd step
      auto odd_slot = [&](auto A_) {
        constexpr int a = decltype(A_)::value;
        const int far = a * kWidth - L::cz(a) * RS - L::cx(a);
        if constexpr (WALL && a != 0) return combo(A_) ? L::opp(a) * kWidth : far;
        else return far;
      };
      R f[Q];
      static_for<0, Q>([&](auto A_) {
        constexpr int a = decltype(A_)::value;
        R v = s[ODD ? odd_slot(A_) : L::opp(a) * kWidth];
        if constexpr (WALL && a != 0) {
          const int c = combo(A_);
          if (c) v = v + args.bb[a][c];
        }
        f[a] = v;
      });
      if (TO && last) {
        R* o = args.dst + (gx + args.pitch * gz);
#pragma unroll
        for (int a = 0; a < Q; ++a) o[a * args.vol] = f[a];
      } else {
        Coef<R> k{};
        moments_coeffs<L, FORCE>(f, args.ph, k);
        if (last) {
          R* o = args.dst + (gx + args.pitch * gz);
          each_coef<L, R>(k, [&](auto I, R& v) { o[decltype(I)::value * args.vol] = v; });
        } else {
          R out[Q];
          post_all<L, R>(k, out);
          static_for<0, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            s[ODD ? odd_slot(A_) : a * kWidth] = out[ODD ? L::opp(a) : a];
          });
        }
      }
    }
  };
  const bool walls = (!args.per_x && (x0 - T <= 0 || x0 + bxa + T >= nx)) ||
                     (!args.per_z && (z0 - T <= 0 || z0 + bza + T >= nz));
  for (int t = 1; t <= T; ++t) {
    __syncthreads();
    if (t & 1) {
      if (walls) step(t, std::true_type{}, std::true_type{});
      else step(t, std::true_type{}, std::false_type{});
    } else {
      if (walls) step(t, std::false_type{}, std::true_type{});
      else step(t, std::false_type{}, std::false_type{});
    }
  }
  static_assert(NC == 6, "2D sets hold six fields");
}

// where set A begins: behind the populations
inline int64_t set_a_at(const Geometry& g) { return int64_t(g.q) * g.vol; }

template <class R>
using K4Kernel = void (*)(const K4Args<R>);

// where: 0 first launch of a run, 1 between, 2 last
template <class R>
K4Kernel<R> k4_kernel(bool force, int where) {
  static const K4Kernel<R> t[2][3] = {
      {k4_steps<R, false, true, false>, k4_steps<R, false, false, false>, k4_steps<R, false, false, true>},
      {k4_steps<R, true, true, false>, k4_steps<R, true, false, false>, k4_steps<R, true, false, true>}};
  return t[force][where];
}

// Launches and tile height of a run of n steps: the least of a launch's time,
// fitted to sweeps of 128 x 96, 301 x 257, 1024^2 and 4096^2 cavities (T = 2 .. 8,
// 8 to 40 rows; within 10 %).  A tile takes about
//   1 + 0.12 rows read + 0.053 rows stepped us (FP64: 0.65 and 2.3)
// with two on an SM, a little less alone, and more where tiles at walls decide
// (fewer than a wave of them).  FP32 picks, us per step: 4096^2 T = 6, 32 rows 97
// (T = 2, 40 rows: 130), 1024^2 T = 8, 32 rows 8.2 (T = 2: 10.6), 301 x 257 T = 8,
// 16 rows 2.0 (8 rows, which put two tiles on an SM: 2.5; T = 2: 3.3); FP64
// 1024^2 T = 2, 16 rows 173 (T = 4: 194, the ring's arithmetic).
struct FlatSplit {
  int64_t launches = 0;
  int bz = 0;
};
FlatSplit split_run(int64_t nx, int64_t nz, int64_t n, int max_rows, bool fp64, int sm_count) {
  FlatSplit best;
  double best_cost = 1e300;
  const double read = fp64 ? 0.65 : 0.12, step = fp64 ? 2.3 : 0.053;
  const double sms = sm_count;
  for (int T = 1; T <= kMaxSteps; ++T) {
    const int64_t launches = 2 * ((n + 2 * T - 1) / (2 * T));
    // an odd n in single steps leaves none for the last launch, which has to
    // write the populations
    if (launches > n) continue;
    const int steps = int((n + launches - 1) / launches);
    const int64_t ntx = (nx + kWidth - 2 * steps - 1) / (kWidth - 2 * steps);
    for (int bz = 8; bz + 2 * steps <= max_rows; bz += 8) {
      const double tiles = double(ntx) * double((nz + bz - 1) / bz);
      const double tile = 1.0 + read * (bz + 2 * steps) + step * steps * (bz + steps - 1);
      const double rounds = tiles <= sms ? 0.9 : std::max(1.7, tiles / (2 * sms) + 0.5);
      const double cost = double(launches) * (3.0 + rounds * tile);
      if (cost < best_cost) {
        best_cost = cost;
        best.launches = launches;
        best.bz = bz;
      }
    }
  }
  return best;
}

// steps of launch i: as even as they come, the longer launches first
int launch_steps(int64_t n, int64_t launches, int64_t i) { return int(n / launches + (i < n % launches ? 1 : 0)); }

template <class R>
cudaError_t flat_run_as(lb_ctx* ctx, int64_t n, bool beside) {
  const Geometry& g = ctx->g;
  const FlatSplit sp = split_run(g.nx, g.nz, n, k4_max_rows<R>(), sizeof(R) == 8, k1_sm_count());
  if (sp.launches < 2) return cudaErrorInvalidValue;
  R* const f = static_cast<R*>(ctx->f);
  R* const set[2] = {f + set_a_at(g), f};
  K4Args<R> a;
  a.ph = make_phys<R>(g);
  a.nx = g.nx;
  a.nz = g.nz;
  a.pitch = g.pitch;
  a.vol = g.vol;
  a.per_x = g.per[0];
  a.per_z = g.per[2];
  for (int i = 0; i < 27; ++i)
    for (int j = 0; j < 8; ++j) a.bb[i][j] = R(0);
  make_bounce_terms<D2Q9, R>(g, a.bb);
  a.bz = sp.bz;
  cudaError_t e = cudaSuccess;
  for (int64_t i = 0; i < sp.launches && e == cudaSuccess; ++i) {
    const bool last = i == sp.launches - 1;
    a.steps = launch_steps(n, sp.launches, i);
    a.bx = kWidth - 2 * a.steps;
    a.ntx = div_up(g.nx, a.bx);
    a.src = i == 0 ? f : set[(i - 1) & 1];
    a.dst = last ? f : set[i & 1];
    const int grid = a.ntx * div_up(g.nz, a.bz);
    const size_t smem = size_t(a.bz + 2 * a.steps) * 9 * kWidth * sizeof(R);
    e = launch_step(k4_kernel<R>(g.has_force, i == 0 ? 0 : last ? 2 : 1), grid, k4_threads<R>(), smem, ctx->stream,
                    !beside && i > 0 && grid <= 2 * k1_sm_count(), a);
  }
  return e;
}

template <class R>
bool configure() {
  for (int force = 0; force < 2; ++force)
    for (int where = 0; where < 3; ++where)
      if (cudaFuncSetAttribute(k4_kernel<R>(force, where), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(kTileSmem)) != cudaSuccess) {
        cudaGetLastError();
        return false;
      }
  return true;
}

}  // namespace

size_t flat_scratch_elems(const Geometry& g, int storage) {
  if (g.lattice != LB_D2Q9 || (storage != LB_F32 && storage != LB_F64)) return 0;
  return size_t(set_a_at(g)) + 6 * size_t(g.vol);
}

bool flat_plan(lb_ctx* ctx) {
  if (ctx->flat_state != 0) return ctx->flat_state > 0;
  ctx->flat_state = -1;
  const size_t need = flat_scratch_elems(ctx->g, ctx->storage) * ctx->real_bytes;
  if (ctx->scheme != LB_SCHEME_FUSED || ctx->g.zlink[0] || ctx->g.zlink[1] || need == 0 || ctx->f_alloc < need)
    return false;
  if (!(ctx->storage == LB_F64 ? configure<double>() : configure<float>())) return false;
  ctx->flat_state = 1;
  return true;
}

cudaError_t flat_run(lb_ctx* ctx, int64_t n, bool beside) {
  const cudaError_t e =
      ctx->storage == LB_F64 ? flat_run_as<double>(ctx, n, beside) : flat_run_as<float>(ctx, n, beside);
  return e == cudaSuccess ? k1_bootstrap(ctx) : e;
}

}  // namespace lbgb

extern "C" int lb_plan_flat(int32_t storage, const int64_t dims[3], int64_t n, int32_t sms, lb_flat_plan_t* out) {
  using namespace lbgb;
  if (!out || !dims || n < 2 || dims[2] != 1) return LB_E_INVAL;
  for (int k = 0; k < 2; ++k)
    if (dims[k] < 1 || dims[k] > (int64_t(1) << 30)) return LB_E_INVAL;
  if (storage != LB_F64 && storage != LB_F32) return LB_E_UNSUPPORTED;
  const bool fp64 = storage == LB_F64;
  const int rows = fp64 ? k4_max_rows<double>() : k4_max_rows<float>();
  const FlatSplit sp = split_run(dims[0], dims[1], n, rows, fp64, sms > 0 ? sms : k1_sm_count());
  out->launches = sp.launches;
  out->steps_first = launch_steps(n, sp.launches, 0);
  out->steps_last = launch_steps(n, sp.launches, sp.launches - 1);
  out->tile_rows = sp.bz;
  out->max_rows = rows;
  return LB_OK;
}
