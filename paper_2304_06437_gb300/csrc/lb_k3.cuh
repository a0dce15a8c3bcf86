// lb_k3.cuh -- the step in moment form, for runs of several steps.
//
// The post-collision set of a node is a quadratic form in c_a whose
// coefficients (lb_collide.cuh: A, B, C, C2) follow from its density, velocity
// and stress (section 3 of the paper: the multline step equation).  Between
// two steps of one lb_step() call a node's state is therefore these n_coef
// values (10 in 3D, 6 in 2D) instead of its q populations:
//
//     coef(x, t+1) = collide( { post_a( coef(x - c_a, t) ) }_a )
//
// A run of n steps is: one pass that turns the populations into coefficients
// in place (k3_enter), n - 1 launches of k3_step from one set of coefficient
// fields into another, and one brick launch that pulls the populations of the
// last step back (k1_leave_step, lb_k1.cuh).  Every arithmetic operation is
// that of the population form, in its order, and the coefficients are kept in
// the arithmetic type, so the populations are bit for bit those of n
// single-step launches.
//
// Why: the population form moves 2 q values per update and is bound by HBM
// (D3Q27 FP32) or by instruction issue close to it (D3Q19 FP32); the moment
// form moves 2 n_coef: 80 instead of 152 / 216 bytes per update for D3Q19 /
// D3Q27 FP32.  It also needs no shell: source and destination differ, so a
// tile reads its one-node halo from the source set (L2 holds what the
// neighbouring tiles read), and nothing is collided twice.  Measured per step
// on one GB300, single-step launches against this form: D3Q19 FP32 512^3 35.2
// -> 63.5 GLUPS (5.1 TB/s, 0.75 of the copy rate), 256^3 31.9 -> 60.3, 32^3
// 24.8 -> 4.3 us; D3Q27 FP32 256^3 25.6 -> 47.0 (0.56); D3Q19 / D3Q27 FP64 96^3
// 2.19 -> 3.17 / 1.10 -> 1.88 (bound by the FP64 rate); D3Q19 FP16 160^3 161 ->
// 72 us (57 GLUPS: the FP32 rate, two roundings a value on top).  What bounds the FP32
// kernels: instruction issue (62 % of the slots) and, without the halo warps'
// part, 71 GLUPS.
//
// Memory: the two sets of coefficient fields live in the population array
// itself -- set A in fields 0 .. n_coef - 1, set B in the n_coef fields after
// it -- and its allocation goes on through the shell buffers (idle meanwhile,
// rebuilt at the end), which hold what 2 n_coef fields exceed q by and the edge
// records below.  16-bit populations are smaller than a set: set B takes their
// place and what follows, set A the n_coef fields after that, and the last
// step goes straight from set A to the populations (POP).
//
// Layout of a launch: a CTA owns a tile of bx x by nodes and sweeps bz planes.
// TMA streams the tile's coefficients plane by plane into a ring of shared
// slots; each node thread evaluates the post-collision set of its node and puts
// the laterally moving populations into a shared window (three buffers).  Halo
// warps fill the one-node ring around the tile, from loads issued a plane ahead:
// with the populations that enter from the neighbouring tiles, or, where the
// tile borders an x or y wall, with the bounce-back values of the wall's own
// nodes, so that the node warps gather without any test for walls.  One split
// barrier per plane: a warp arrives once its part of a window is written and
// waits when it needs the whole.  (Two nodes a thread in packed FP32x2
// arithmetic measured slower.)
#pragma once

#include "lb_k1.cuh"

namespace lbgb {

// Edge records: the coefficients of the nodes in the first (side 0) and last
// (side 1) column of every tile, NC consecutive values a node and consecutive
// along y, which the neighbouring tiles' ring columns are read from.  (Read
// from the fields, every value is a sector of its own; D3Q19 64 x 8 tiles with
// little L1 cache beside their shared memory: 51.9 against 59.9 GLUPS.)
// Record of row r = y + ny z of tile column tI.
LB_HD inline int64_t k3_edge(int side, int tI, int ntx, int64_t rows, int64_t r) {
  return (int64_t(side) * ntx + tI) * rows + r;
}

template <class R>
struct K3Args {
  Phys<R> ph;
  int nx, ny, nz;
  int64_t pitch, vol;
  int per[3];
  int bz, ntx, nty, ntz;  // sweep length, tiles along x and y, bricks along z
  const R* src;           // coefficient fields read, and
  R* dst;                 // written: field i at + i * vol
  const R* esrc;          // edge records of the two sets (see k3_edge)
  R* edst;
  int* status;
  uint32_t vol32;         // vol / 32 (rows are padded to 32 elements)
  void* pop;              // populations written instead of dst (POP)
  R bb[27][8];
};

// the direction along +-z (sign) that does not move laterally
template <class L, int sign>
LB_HD constexpr int nonlateral_dir() {
  for (int a = 0; a < L::Q; ++a)
    if (L::cx(a) == 0 && L::cy(a) == 0 && L::cz(a) == sign) return a;
  return -1;
}

template <class L, class R, int BX, int BY, int NS, int MINB>
struct K3Shape {
  static constexpr int Q = L::Q;
  static constexpr int NC = n_coef<L>();
  static constexpr int NYF = count_dirs<L>(1, 1);
  static constexpr int PY = NYF > 0 ? 1 : 0;
  static constexpr int NTM = BX * BY;      // node threads
  static constexpr int WY = BY + 2 * PY;   // window rows
  // Window of one direction: rows of the tile and its ring.  A direction with
  // cx = 0 needs no ring along x: rows of BX values.  The others have rows of
  // BX + 2, column xl of the tile (-1 .. BX) at xl + 1.
  LB_HD static constexpr int row(int a) { return L::cx(a) == 0 ? BX : BX + 2; }
  // position of the tile's column xl in a row of a moving direction
  LB_HD static constexpr int col(int xl) { return xl + 1; }
  LB_HD static constexpr int off(int a) {
    int n = 0;
    for (int b = 0; b < a; ++b)
      if (is_lateral<L>(b)) n += WY * row(b);
    return n;
  }
  // halo threads: south and north rows (one per column), then the
  // west and east columns with the corners, each column in warps of its own
  // (a warp of two faces runs both in turn, and is then what the others wait for)
  static constexpr int HROW = NYF > 0 ? 2 * BX : 0;
  static constexpr int HCOL = NYF > 0 ? (WY + 31) / 32 * 32 : 16;
  static constexpr int HWARPS = (HROW + 2 * HCOL) / 32;
  static constexpr int NT = NTM + 32 * HWARPS;
  static constexpr int NWARPS = NT / 32;
  static constexpr int SLOTN = NC * BY * BX;  // elements of one plane of the tile
  static constexpr size_t WIN = align128(size_t(off(Q)) * sizeof(R));
  static constexpr size_t OFF_WIN = align128(size_t(NS) * SLOTN * sizeof(R));
  static constexpr size_t SMEM_CAP = (size_t(228) * 1024) / MINB - 1024;
  static constexpr int NW = 3;  // window buffers
  // the halo threads' coefficients, HD planes deep
  static constexpr int HD = 4;
  static constexpr size_t HSTAGE = size_t(NC) * (HROW + 2 * HCOL) * sizeof(R);
  static constexpr size_t OFF_HALO = OFF_WIN + NW * WIN;
  static constexpr size_t OFF_BAR = align128(OFF_HALO + HD * HSTAGE);
  static constexpr size_t SMEM = OFF_BAR + align128((NS + NW) * sizeof(uint64_t));
  static_assert(SMEM <= SMEM_CAP, "shared memory of the shape exceeds its share of the SM");
  static_assert(NTM % 32 == 0 && NT <= 1024, "whole warps");
  static_assert(BY == 1 || NYF > 0, "a 2D tile has one internal row");
  static_assert(HROW % 32 == 0, "a halo warp holds rows or columns, not both");
};

// a node's coefficients as one record (16- or 8-byte stores)
template <class L, class R>
LB_DEV void put_record(Coef<R>& k, R* e) {
  using R2 = typename std::conditional<sizeof(R) == 4, float2, double2>::type;
  R rec[n_coef<L>()];
  each_coef<L, R>(k, [&](auto I, R& v) { rec[decltype(I)::value] = v; });
#pragma unroll
  for (int i = 0; i < n_coef<L>(); i += 2) reinterpret_cast<R2*>(e)[i / 2] = R2{rec[i], rec[i + 1]};
}

// One step of one brick (tile column tI, tJ, sweep tK): src -> dst, or (POP)
// src -> populations, the last step of a run whose set A lies behind them.
template <class L, class S, class R, int BX, int BY, int NS, bool FORCE, int MINB, bool POP>
__device__ __forceinline__ void k3_brick(const CUtensorMap* tmap_p, const K3Args<R>& args, const int tI, const int tJ,
                                         const int tK) {
  using Sh = K3Shape<L, R, BX, BY, NS, MINB>;
  constexpr int Q = L::Q, NC = Sh::NC, NTM = Sh::NTM, NYF = Sh::NYF, PY = Sh::PY;
  constexpr int WY = Sh::WY, HROW = Sh::HROW, NW = Sh::NW;
  constexpr int RM = BX + 2;  // row of a moving direction
  constexpr int WSTRIDE = int(Sh::WIN / sizeof(R));
  constexpr int SLOTN = Sh::SLOTN;

  extern __shared__ __align__(128) unsigned char smem[];
  R* slots = reinterpret_cast<R*>(smem);
  R* win0 = reinterpret_cast<R*>(smem + Sh::OFF_WIN);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Sh::OFF_BAR);
  uint64_t* wbars = bars + NS;

  const int tid = threadIdx.x;
  const bool is_main = tid < NTM;
  const int nx = args.nx, ny = args.ny, nz = args.nz;
  const int x0 = tI * BX, y0 = tJ * BY, z0 = tK * args.bz;
  const int bxa = min(BX, nx - x0), bya = min(BY, ny - y0);
  const int z1 = min(z0 + args.bz, nz);
  const int64_t plane = args.pitch * ny;  // elements between planes of a field

  // planes z0 - 1 .. z1 are needed; the outer two only where they exist
  const bool nbD = z0 > 0 || args.per[2];
  const bool nbU = z1 < nz || args.per[2];
  const int zb = nbD ? z0 - 1 : z0;  // first and last plane produced
  const int ze = nbU ? z1 : z1 - 1;
  auto zwrap = [&](int z) { return z < 0 ? z + nz : (z >= nz ? z - nz : z); };

  // faces of the tile at a wall
  const bool wallW = x0 == 0 && !args.per[0], wallE = x0 + bxa == nx && !args.per[0];
  const bool wallS = y0 == 0 && !args.per[1], wallN = y0 + bya == ny && !args.per[1];

  int issued = 0;  // planes whose load was issued (thread 0's count)
  // thread 0: load plane zb + k into slot k % NS
  auto load_plane = [&](int k) {
    uint64_t* bar = &bars[k % NS];
    mbar_arrive_expect_tx(bar, uint32_t(SLOTN * sizeof(R)));
    tma_load_4d(slots + (k % NS) * SLOTN, tmap_p, x0, y0, zwrap(zb + k), 0, bar);
    ++issued;
  };
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(&bars[s], 1);
    for (int s = 0; s < NW; ++s) mbar_init(&wbars[s], Sh::NWARPS);
    fence_barrier_init();
  }
  // what came before may still run up to here (launch_step); the next launch
  // may be brought in beside this one
  grid_wait();
  grid_release();
  if (tid == 0)
    for (int s = 0; s < NS && zb + s <= ze; ++s) load_plane(s);
  __syncthreads();

  // a thread whose bounded wait ran out stops waiting and runs the sweep to its
  // end (on undefined values, like the rest of the launch), so that every warp
  // still arrives at every barrier
  bool dead = false;
  // windows: plane zb + k uses buffer k % NW.  A warp arrives when it has put
  // its populations of a plane into the window and waits just before it
  // gathers them, with the gather and collision of the plane before in between.
  // A warp that has passed plane k's barrier knows that every warp has gathered
  // plane k - 2, so it may fill the buffer of plane k + NW - 2.
  auto window_ready = [&](int k) {
    __syncwarp();
    if (tid % 32 == 0) mbar_arrive(&wbars[k % NW]);
  };
  auto window_wait = [&](int k) {
    if (!dead && !mbar_wait_bounded(&wbars[k % NW], (k / NW) & 1, kWaitLimitNs)) dead = true;
  };
  auto slot_wait = [&](int k) {
    if (!dead && !mbar_wait_bounded(&bars[k % NS], (k / NS) & 1, kWaitLimitNs)) dead = true;
  };

  if (!is_main) {
    // ------------------------------------------------------------ halo warps
    // face crossed (0 W, 1 E, 2 S, 3 N); kind 0 nothing, 1 a neighbouring
    // node whose populations enter, 2 a node at the wall whose own come back
    const int hid = tid - NTM;
    using i0 = std::integral_constant<int, 0>;
    using i1 = std::integral_constant<int, 1>;
    using im = std::integral_constant<int, -1>;

    // face, kind, the column xl and window row r of the ring cell (kind 2: the
    // node's own column, and r the row beyond the wall for rows); the node (kind
    // 2); its coefficients in plane 0 (rows: in the fields, columns: an edge record)
    auto run = [&](auto col_tag, const int face, const int kind, const int xl, const int r, const int sx,
                   const int sy, const R* const p0) {
      constexpr bool COL = decltype(col_tag)::value;
      // plane zb + p is copied to stage p % HD of this thread's own shared
      // memory, HD - 2 planes ahead (a plane's time is about a loaded memory
      // latency: with loads one plane ahead the whole CTA waited for them)
      constexpr int HD = Sh::HD, HT = COL ? 2 * Sh::HCOL : HROW;
      using R2 = typename std::conditional<sizeof(R) == 4, float2, double2>::type;
      unsigned char* const stage0 = smem + Sh::OFF_HALO + (COL ? size_t(HD) * NC * HROW * sizeof(R) : 0);
      const int ht = COL ? hid - HROW : hid;
      auto fetch = [&](int p) {
        const int z = zb + p;
        if (kind != 0 && z <= ze) {
          if constexpr (COL) {
            const R2* g = reinterpret_cast<const R2*>(p0 + int64_t(ny) * NC * zwrap(z));
            R2* h = reinterpret_cast<R2*>(stage0) + (p % HD) * (NC / 2) * HT + ht;
#pragma unroll
            for (int i = 0; i < NC / 2; ++i) cp_async<sizeof(R2)>(h + i * HT, g + i);
          } else {
            const char* g = reinterpret_cast<const char*>(p0 + plane * zwrap(z));
            const uint32_t v32 = args.vol32;
            R* h = reinterpret_cast<R*>(stage0) + (p % HD) * NC * HT + ht;
#pragma unroll
            for (int i = 0; i < NC; ++i)
              cp_async<sizeof(R)>(h + i * HT, g + uint64_t(v32) * uint32_t(i * 32 * sizeof(R)));
          }
        }
        cp_async_commit();
      };
      auto coef_of = [&](int p) {
        R h[NC];
        if constexpr (COL) {
          const R2* hs = reinterpret_cast<const R2*>(stage0) + (p % HD) * (NC / 2) * HT + ht;
#pragma unroll
          for (int i = 0; i < NC; i += 2) {
            const R2 v = hs[i / 2 * HT];
            h[i] = v.x;
            h[i + 1] = v.y;
          }
        } else {
          const R* hs = reinterpret_cast<const R*>(stage0) + (p % HD) * NC * HT + ht;
#pragma unroll
          for (int i = 0; i < NC; ++i) h[i] = hs[i * HT];
        }
        Coef<R> k;
        each_coef<L, R>(k, [&](auto I, R& v) { v = h[decltype(I)::value]; });
        return k;
      };
      // bounce-back values of the node's descending links, for the next window
      R held[Q];
#pragma unroll
      for (int a = 0; a < Q; ++a) held[a] = R(0);
      // sides the node touches: bit 0 low, bit 1 high
      const int y_walls = args.per[1] ? 0 : (sy == 0 ? 1 : 0) | (sy == ny - 1 ? 2 : 0);
      const int x_walls = args.per[0] ? 0 : (sx == 0 ? 1 : 0) | (sx == nx - 1 ? 2 : 0);

      auto produce = [&](int p, auto AX, auto SG) {
        constexpr int ax = decltype(AX)::value, sg = decltype(SG)::value;
        R* win = win0 + (p % NW) * WSTRIDE;
        if (kind == 1) {
          const Coef<R> k = coef_of(p);
          static_for<0, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            if constexpr (comp<L>(ax, a) == sg) {
              R v = post<L, R, a>(k);
              R* w = win + Sh::off(a) + r * Sh::row(a);
              if constexpr (L::cx(a) == 0) w[xl] = v;
              else w[Sh::col(xl)] = v;
            }
          });
        } else if (kind == 2) {
          const Coef<R> k = coef_of(p), kn = coef_of(p + 1);
          static_for<0, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
            if constexpr (comp<L>(ax, a) == sg) {
              // the link of this node through the wall: the node's own opposite
              // population of the destination plane, c + cz
              auto bounce = [&](const Coef<R>& kk) {
                int cb = 0;
                if constexpr (cx == 1) cb |= x_walls & 1;
                if constexpr (cx == -1) cb |= x_walls >> 1;
                if constexpr (cy == 1) cb |= (y_walls & 1) << 1;
                if constexpr (cy == -1) cb |= y_walls & 2;
                return post<L, R, L::opp(a)>(kk) + args.bb[a][cb];
              };
              R v;
              if constexpr (cz == 0) v = bounce(k);
              else if constexpr (cz == 1) v = bounce(kn);
              else v = held[a];
              if constexpr (cz == -1) held[a] = bounce(k);
              R* w = win + Sh::off(a) + (ax == 1 ? r : r - cy) * Sh::row(a);
              if constexpr (cx == 0) w[xl] = v;
              else w[Sh::col(xl - cx)] = v;
            }
          });
        }
      };
      for (int p = 0; p < HD - 1; ++p) fetch(p);
      for (int p = 0; p <= ze - zb; ++p) {
        // into the stage plane p - 1 was read from; planes up to p + 1 landed
        fetch(p + HD - 1);
        cp_async_wait<HD - 2>();
        if (face == 0) produce(p, i0{}, i1{});
        else if (face == 1) produce(p, i0{}, im{});
        if constexpr (NYF > 0) {
          if (face == 2) produce(p, i1{}, i1{});
          else if (face == 3) produce(p, i1{}, im{});
        }
        window_ready(p);
        // plane p + 1's buffer must be free (see window_ready above)
        if (p + 3 - NW >= 0) window_wait(p + 3 - NW);
      }
    };

    if (hid < HROW) {
      const int face = hid < BX ? 2 : 3;
      const int xl = hid % BX;
      const bool wall = face == 2 ? wallS : wallN;
      int sy = face == 2 ? y0 - 1 : y0 + bya;
      if (wall) sy = face == 2 ? y0 : y0 + bya - 1;  // the wall's own row
      else sy = sy < 0 ? sy + ny : (sy >= ny ? sy - ny : sy);
      run(std::false_type{}, face, xl < bxa ? (wall ? 2 : 1) : 0, xl, face == 2 ? 0 : bya + 1, x0 + xl, sy,
          args.src + (x0 + xl) + args.pitch * sy);
    } else {
      const int k = hid - HROW;
      const int r = k % Sh::HCOL, yl = r - PY;
      const int face = k < Sh::HCOL ? 0 : 1;
      const bool wall = face == 0 ? wallW : wallE;
      // the neighbouring tile's last or first column, or at a wall this tile's
      // own first or last
      const int side = wall ? face : 1 - face;
      const int tc = wall ? tI : (face == 0 ? (tI > 0 ? tI : args.ntx) - 1 : (tI + 1 < args.ntx ? tI + 1 : 0));
      int sy = y0 + yl;
      int kind = r < WY ? (wall ? 2 : 1) : 0;
      if (wall) {
        if (yl < 0 || yl >= bya) kind = 0;
      } else {
        if (yl > bya - 1 + PY) kind = 0;
        // a corner beyond a y wall belongs to that wall's nodes
        if (sy < 0 || sy >= ny) {
          if (args.per[1]) sy = sy < 0 ? sy + ny : sy - ny;
          else kind = 0;
        }
      }
      if (kind == 0) sy = 0;
      // the ring column, or at a wall the column of the node itself
      const int xl = face == 0 ? (wall ? 0 : -1) : (wall ? bxa - 1 : bxa);
      run(std::true_type{}, face, kind, xl, r, x0 + xl, sy,
          args.esrc + k3_edge(side, tc, args.ntx, int64_t(ny) * nz, sy) * NC);
    }
    if (dead) atomicExch(args.status, LB_E_TIMEOUT);
    return;
  }

  // -------------------------------------------------------------- node warps
  const int i = tid % BX, ty = tid / BX;
  const int x = x0 + i, y = y0 + ty;
  const bool active = i < bxa && ty < bya;
  const bool z_walls = !args.per[2];
  // this thread's place in the rows of the two kinds of directions
  const int b0 = (ty + PY) * BX + i;
  const int bm = (ty + PY) * RM + i;
  R* const out0 = args.dst + x + args.pitch * y;
  // edge records this thread writes: of the tile's first and last columns
  const bool west = i == 0, east = i < bxa && i + 1 >= bxa;
  R* const edge0 = args.edst + k3_edge(west ? 0 : 1, tI, args.ntx, int64_t(ny) * nz, y) * NC;
  constexpr int zm = nonlateral_dir<L, -1>(), zp = nonlateral_dir<L, 1>();

  auto put = [&](R* win, auto A_, R v) {
    constexpr int a = decltype(A_)::value;
    if constexpr (L::cx(a) == 0) win[Sh::off(a) + b0] = v;
    else win[Sh::off(a) + bm + 1] = v;
  };
  // the value of direction a at the thread's node shifted by (-dx, -dy)
  auto get = [&](const R* win, auto A_, auto DX, auto DY) -> R {
    constexpr int a = decltype(A_)::value, dx = decltype(DX)::value, dy = decltype(DY)::value;
    if constexpr (L::cx(a) == 0) {
      return win[Sh::off(a) + b0 - dy * BX];
    } else {
      const R* w = win + Sh::off(a) + bm - dy * RM;
      return w[1 - dx];
    }
  };

  // collide plane c = zb + k: the laterally moving populations go to the window, the
  // others to their destinations (rest: plane c, -z: c - 1, +z: c + 1)
  auto produce = [&](int k, R* win, R& rest, R& down, R& up) {
    slot_wait(k);
    if (active) {
      const R* sl = slots + (k % NS) * SLOTN + tid;
      Coef<R> kc;
      each_coef<L, R>(kc, [&](auto I, R& v) { v = sl[decltype(I)::value * (BX * BY)]; });
      rest = post<L, R, 0>(kc);
      static_for<1, Q>([&](auto A_) {
        constexpr int a = decltype(A_)::value;
        constexpr int b = L::opp(a);
        if constexpr (leading_sign<L>(a) == 1) {
          R fa, fb;
          post_pair<L, a>(kc, fa, fb);
          if constexpr (is_lateral<L>(a)) {
            put(win, A_, fa);
            put(win, std::integral_constant<int, b>{}, fb);
          } else {
            static_assert(a == zp && b == zm, "the pair along z");
            up = fa;
            down = fb;
          }
        }
      });
    }
  };

  // gathered populations of three destination planes; the roles of the sets
  // are permuted at compile time
  R G[3][Q];
  produce(0, win0, G[1][0], G[0][zm], G[2][zp]);
  window_ready(0);
  window_wait(0);

  // trip t, plane g = zb + 3 t + k
  auto sweep_plane = [&](const int t, auto K) {
    constexpr int k = decltype(K)::value;
    const int g = zb + 3 * t + k;
    const int kc = 3 * t + k + 1;  // plane c's index
    R(&G0)[Q] = G[k % 3];          // destination plane g - 1
    R(&G1)[Q] = G[(k + 1) % 3];    // g
    R(&G2)[Q] = G[(k + 2) % 3];    // g + 1
    const int c = g + 1;
    const R* win_g = win0 + (kc - 1) % NW * WSTRIDE;
    R* win_c = win0 + kc % NW * WSTRIDE;
    R up_c = R(0);  // plane c's +z population: of plane c + 1, whose set is G0
    const R down_g = G0[zm], up_g = G2[zp];  // this node's own, for a z wall's bounce-back
    if (c <= ze) {
      produce(kc, win_c, G2[0], G1[zm], up_c);
      window_ready(kc);
    }

    if (active) {
      if (g <= ze) {
        static_for<1, Q>([&](auto A_) {
          constexpr int a = decltype(A_)::value;
          constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
          if constexpr (is_lateral<L>(a)) {
            const R v = get(win_g, A_, std::integral_constant<int, cx>{}, std::integral_constant<int, cy>{});
            if constexpr (cz == -1) G0[a] = v;
            if constexpr (cz == 0) G1[a] = v;
            if constexpr (cz == 1) G2[a] = v;
          }
        });
        // halfway bounce-back at a z wall
        if (z_walls && (g == 0 || g == nz - 1)) {
          const bool z_lo = g == 0, z_hi = g == nz - 1;
          static_for<1, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
            if constexpr (cz != 0) {
              if (cz == 1 ? z_lo : z_hi) {
                constexpr int oa = L::opp(a);
                R v;
                if constexpr (is_lateral<L>(oa))
                  v = get(win_g, std::integral_constant<int, oa>{}, std::integral_constant<int, 0>{},
                          std::integral_constant<int, 0>{});
                else
                  v = oa == zm ? down_g : up_g;
                int cb = 4;
                if constexpr (cy == 1) cb |= y == 0 && !args.per[1] ? 2 : 0;
                if constexpr (cy == -1) cb |= y == ny - 1 && !args.per[1] ? 2 : 0;
                if constexpr (cx == 1) cb |= x == 0 && !args.per[0] ? 1 : 0;
                if constexpr (cx == -1) cb |= x == nx - 1 && !args.per[0] ? 1 : 0;
                G1[a] = v + args.bb[a][cb];
              }
            }
          });
        }
      }
      // plane g - 1 is complete: collide it
      const int zd = g - 1;
      if (zd >= z0) {
        if constexpr (POP) {
          S* o = static_cast<S*>(args.pop) + (x + args.pitch * y + plane * zd);
          static_for<0, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            o[a * args.vol] = store_as<S, R>(G0[a]);
          });
        } else {
          R fr[Q];
          static_for<0, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            fr[a] = round_to_storage<S, R>(G0[a]);
          });
          Coef<R> kc2;
          moments_coeffs<L, FORCE>(fr, args.ph, kc2);
          char* o = reinterpret_cast<char*>(out0 + plane * zd);
          const uint32_t v32 = args.vol32;
          each_coef<L, R>(kc2, [&](auto I, R& v) {
            *reinterpret_cast<R*>(o + uint64_t(v32) * uint32_t(decltype(I)::value * 32 * sizeof(R))) = v;
          });
          if (west || east) {
            R* e = edge0 + int64_t(ny) * NC * zd;
            put_record<L>(kc2, e);
            // a tile of one column is both
            if (west && east) put_record<L>(kc2, e + int64_t(args.ntx) * ny * nz * NC);
          }
        }
      }
    }
    G0[zp] = up_c;
    if (c <= ze) {
      window_wait(kc);
      // every thread has read plane c's slot
      if (tid == 0 && !dead && c + NS <= ze) load_plane(kc + NS);
    }
  };
  // the slot of plane zb is free once its window is complete
  if (tid == 0 && !dead && zb + NS <= ze) load_plane(NS);
  // gathers planes zb .. ze, completes planes z0 .. z1 - 1 (the last trip,
  // g = z1, only completes where plane z1 does not exist)
  const int trips = z1 - zb + 1;
  for (int t = 0; 3 * t < trips; ++t) {
    sweep_plane(t, std::integral_constant<int, 0>{});
    if (3 * t + 1 >= trips) break;
    sweep_plane(t, std::integral_constant<int, 1>{});
    if (3 * t + 2 >= trips) break;
    sweep_plane(t, std::integral_constant<int, 2>{});
  }
  if (dead) {
    atomicExch(args.status, LB_E_TIMEOUT);
    if (tid == 0) {
      // copies still in flight may write this CTA's shared memory: wait for
      // them (bounded)
      bool drained = true;
      for (int k = issued - NS < 0 ? 0 : issued - NS; k < issued; ++k)
        drained &= mbar_wait_bounded(&bars[k % NS], (k / NS) & 1, kWaitLimitNs);
      if (!drained) atomicExch(args.status, LB_E_ABANDONED);
    }
  }
}

template <class L, class S, class R, int BX, int BY, int NS, bool FORCE, int MINB, bool POP = false>
__global__ void __launch_bounds__(K3Shape<L, R, BX, BY, NS, MINB>::NT, MINB)
    k3_step(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ K3Args<R> args) {
  const int b = blockIdx.x;
  k3_brick<L, S, R, BX, BY, NS, FORCE, MINB, POP>(&tmap, args, b % args.ntx, (b / args.ntx) % args.nty,
                                                  b / (args.ntx * args.nty));
}

// Populations -> coefficient fields and edge records, node by node (each thread
// reads all of its node's populations before it writes, so the fields may lie
// in the population array).  bx: the tile width the edge records are for.
template <class L, class S, class R, bool FORCE>
__global__ void __launch_bounds__(256)
    k3_enter(const S* f, R* dst, R* edst, int64_t vol, int nx, int64_t rows, int pitch, int bx, Phys<R> ph) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < vol; i += int64_t(gridDim.x) * blockDim.x) {
    // rows are whole 32-element segments; the padding of a row stays zero
    const uint32_t segs = uint32_t(pitch >> 5), seg = uint32_t(i >> 5), row = seg / segs;
    const int x = int((seg - row * segs) * 32 + uint32_t(i & 31));
    if (x >= nx) continue;
    R fr[L::Q];
    static_for<0, L::Q>([&](auto A_) {
      constexpr int a = decltype(A_)::value;
      fr[a] = load_as<S, R>(f[a * vol + i]);
    });
    Coef<R> kc;
    moments_coeffs<L, FORCE>(fr, ph, kc);
    each_coef<L, R>(kc, [&](auto I, R& v) { dst[decltype(I)::value * vol + i] = v; });
    const int tI = x / bx, xl = x - tI * bx, ntx = (nx + bx - 1) / bx;
    constexpr int NC = n_coef<L>();
    if (xl == 0) put_record<L>(kc, edst + k3_edge(0, tI, ntx, rows, row) * NC);
    if (xl == bx - 1 || x == nx - 1) put_record<L>(kc, edst + k3_edge(1, tI, ntx, rows, row) * NC);
  }
}

}  // namespace lbgb
