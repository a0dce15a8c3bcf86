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
// tile reads its one-node halo straight from the source fields (L2 holds what
// the neighbouring tiles read), and nothing is collided twice.
//
// Memory: the two sets of coefficient fields live in the population array
// itself -- set A in fields 0 .. n_coef - 1, set B in the n_coef fields after
// field q/2 -- which the allocation extends to 2 n_coef fields where q is
// smaller (the shell buffers, idle meanwhile, are that extension in 3D).
//
// Layout of a launch: a CTA owns a tile of bx x by nodes and sweeps bz planes.
// TMA streams the tile's coefficients plane by plane into a ring of shared
// slots; each node thread evaluates its post-collision set and puts the
// laterally moving populations into a shared window (three buffers); halo
// warps do the same for the one-node ring around the tile, from loads issued
// one plane ahead, and only for the populations that enter the tile.  One
// split barrier per plane: a warp arrives once its part of a window is
// written and waits when it needs the whole.
#pragma once

#include "lb_k1.cuh"

namespace lbgb {

template <class R>
struct K3Args {
  Phys<R> ph;
  int nx, ny, nz;
  int64_t pitch, vol;
  int per[3];
  int bz, ntx, nty, ntz;  // sweep length, tiles along x and y, bricks along z
  const R* src;           // coefficient fields read, and
  R* dst;                 // written: field i at + i * vol
  int* status;
  uint32_t vol32;         // vol / 32 (rows are padded to 32 elements)
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
  static constexpr int NTM = BX * BY;  // threads that own a node
  static constexpr int NYF = count_dirs<L>(1, 1);
  static constexpr int NLAT = n_lateral<L>();
  static constexpr int PY = NYF > 0 ? 1 : 0;
  static constexpr int WX = BX + 2;
  static constexpr int WY = BY + 2 * PY;
  static constexpr int WPLANE = WX * WY;
  // halo entries, one per thread of the halo warps: south and north rows
  // (whole warps), then the west and east columns with the corners
  static constexpr int HROW = NYF > 0 ? 2 * BX : 0;
  static constexpr int HWARPS = (HROW + 2 * WY + 31) / 32;
  static constexpr int NT = NTM + 32 * HWARPS;
  static constexpr size_t SLOT = size_t(NC) * BY * BX * sizeof(R);
  static constexpr size_t WIN = align128(size_t(NLAT) * WPLANE * sizeof(R));
  static constexpr size_t OFF_WIN = align128(NS * SLOT);
  static constexpr size_t OFF_BAR = OFF_WIN + 3 * WIN;
  static constexpr size_t SMEM = OFF_BAR + align128((NS + 3) * sizeof(uint64_t));
  static constexpr int NWARPS = NT / 32;
  static constexpr size_t SMEM_CAP = (size_t(228) * 1024) / MINB - 1024;
  static_assert(SMEM <= SMEM_CAP, "shared memory of the shape exceeds its share of the SM");
  static_assert(NTM % 32 == 0 && NT <= 1024, "whole warps");
  static_assert(BY == 1 || NYF > 0, "a 2D tile has one internal row");
};

// One step of one brick (tile column tI, tJ, sweep tK): src -> dst.
template <class L, class S, class R, int BX, int BY, int NS, bool FORCE, int MINB>
__device__ __forceinline__ void k3_brick(const CUtensorMap* tmap_p, const K3Args<R>& args, const int tI, const int tJ,
                                         const int tK) {
  using Sh = K3Shape<L, R, BX, BY, NS, MINB>;
  constexpr int Q = L::Q, NC = Sh::NC, NTM = Sh::NTM, NYF = Sh::NYF, PY = Sh::PY;
  constexpr int WX = Sh::WX, WY = Sh::WY, WPLANE = Sh::WPLANE, HROW = Sh::HROW;
  constexpr int WSTRIDE = int(Sh::WIN / sizeof(R));

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

  int issued = 0;  // planes whose load was issued (thread 0's count)
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(&bars[s], 1);
    for (int s = 0; s < 3; ++s) mbar_init(&wbars[s], Sh::NWARPS);
    fence_barrier_init();
    prefetch_tmap(tmap_p);
    for (int s = 0; s < NS && zb + s <= ze; ++s, ++issued) {
      mbar_arrive_expect_tx(&bars[s], static_cast<uint32_t>(Sh::SLOT));
      tma_load_4d(slots + size_t(s) * NC * BY * BX, tmap_p, x0, y0, zwrap(zb + s), 0, &bars[s]);
    }
  }
  __syncthreads();

  // a thread whose bounded wait ran out stops waiting and runs the sweep to its
  // end (on undefined values, like the rest of the launch), so that every warp
  // still arrives at every barrier
  bool dead = false;
  // windows: plane zb + k uses buffer k % 3.  A warp arrives when it has put its
  // populations of a plane into the window and waits just before it gathers
  // them, with the gather and collision of the plane before in between.  A
  // warp that has passed plane k's barrier knows that every warp has gathered
  // plane k - 2, so with three buffers it may fill plane k + 1's.
  auto window_ready = [&](int k) {
    __syncwarp();
    if (tid % 32 == 0) mbar_arrive(&wbars[k % 3]);
  };
  auto window_wait = [&](int k) {
    if (!dead && !mbar_wait_bounded(&wbars[k % 3], (k / 3) & 1, kWaitLimitNs)) dead = true;
  };

  if (!is_main) {
    // ------------------------------------------------------------ halo warps
    const int hid = tid - NTM;
    int sx = 0, sy = 0, cell = 0, face = -1;  // source node, window cell, face crossed
    if (hid < HROW) {
      const int i = hid % BX;
      face = hid < BX ? 2 : 3;
      sx = x0 + i;
      sy = face == 2 ? y0 - 1 : y0 + bya;
      cell = (face == 2 ? 0 : bya + 1) * WX + 1 + i;
      if (i >= bxa) face = -1;
    } else if (hid < HROW + 2 * WY) {
      const int k = hid - HROW;
      const int r = k % WY;
      face = k < WY ? 0 : 1;
      sx = face == 0 ? x0 - 1 : x0 + bxa;
      sy = y0 - PY + r;
      cell = r * WX + (face == 0 ? 0 : bxa + 1);
      if (r >= bya + 2 * PY) face = -1;
    }
    // periodic images; beyond a wall nothing is ever pulled from
    if (sx < 0 || sx >= nx) {
      if (args.per[0]) sx = sx < 0 ? sx + nx : sx - nx;
      else face = -1;
    }
    if (sy < 0 || sy >= ny) {
      if (args.per[1]) sy = sy < 0 ? sy + ny : sy - ny;
      else face = -1;
    }
    const R* p0 = args.src + sx + args.pitch * sy;
    R h[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) h[i] = R(0);
    auto fetch = [&](int z) {
      if (face >= 0 && z <= ze) {
        const R* p = p0 + plane * zwrap(z);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          h[i] = *p;
          p += args.vol;
        }
      }
    };
    auto produce = [&](int c) {
      R* win = win0 + ((c - zb) % 3) * WSTRIDE + cell;
      Coef<R> k;
      each_coef<L, R>(k, [&](auto I, R& v) { v = h[decltype(I)::value]; });
      fetch(c + 1);
      auto put = [&](auto AX, auto SG) {
        constexpr int ax = decltype(AX)::value, sg = decltype(SG)::value;
        static_for<0, Q>([&](auto A_) {
          constexpr int a = decltype(A_)::value;
          if constexpr (comp<L>(ax, a) == sg) win[lat_index<L>(a) * WPLANE] = post<L, R, a>(k);
        });
      };
      using i0 = std::integral_constant<int, 0>;
      using i1 = std::integral_constant<int, 1>;
      using im = std::integral_constant<int, -1>;
      if (face == 0) put(i0{}, i1{});
      else if (face == 1) put(i0{}, im{});
      if constexpr (NYF > 0) {
        if (face == 2) put(i1{}, i1{});
        else if (face == 3) put(i1{}, im{});
      }
    };
    fetch(zb);
    for (int c = zb; c <= ze; ++c) {
      produce(c);
      window_ready(c - zb);
      window_wait(c - zb);
    }
    if (dead) atomicExch(args.status, LB_E_TIMEOUT);
    return;
  }

  // -------------------------------------------------------------- node warps
  const int tx = tid % BX, ty = tid / BX;
  const int x = x0 + tx, y = y0 + ty;
  const bool active = tx < bxa && ty < bya;
  const bool bxlo = x == 0 && !args.per[0];
  const bool bxhi = x == nx - 1 && !args.per[0];
  const bool bylo = y == 0 && !args.per[1];
  const bool byhi = y == ny - 1 && !args.per[1];
  const bool xy_wall = bxlo || bxhi || bylo || byhi;
  const bool z_walls = !args.per[2];
  const int wbase = (ty + PY) * WX + (tx + 1);
  R* const out0 = args.dst + x + args.pitch * y;

  constexpr int zm = nonlateral_dir<L, -1>(), zp = nonlateral_dir<L, 1>();
  // collide plane c = zb + k: the laterally moving populations go to the window, the
  // others to their destinations (rest: plane c, -z: c - 1, +z: c + 1)
  auto produce = [&](int k, R& rest, R& down, R& up) {
    const int slot = k % NS;
    if (!dead && !mbar_wait_bounded(&bars[slot], (k / NS) & 1, kWaitLimitNs)) dead = true;
    if (active) {
      R* win = win0 + (k % 3) * WSTRIDE + wbase;
      const R* sl = slots + size_t(slot) * NC * NTM + tid;
      Coef<R> kc;
      each_coef<L, R>(kc, [&](auto I, R& v) { v = sl[decltype(I)::value * NTM]; });
      rest = post<L, R, 0>(kc);
      static_for<0, n_pairs<L>()>([&](auto P) {
        constexpr int a = pair_first<L>(decltype(P)::value);
        constexpr int b = L::opp(a);
        constexpr R w = R(weight<L>(a));
        R even, wodd;
        post_parts<L, R, a>(kc, even, wodd);
        const R fa = fma_r(w, even, wodd), fb = fma_r(w, even, -wodd);
        if constexpr (is_lateral<L>(a)) {
          win[lat_index<L>(a) * WPLANE] = fa;
          win[lat_index<L>(b) * WPLANE] = fb;
        } else {
          (a == zp ? up : down) = fa;
          (b == zp ? up : down) = fb;
        }
      });
    }
  };

  // load plane zb + k + NS into the slot of plane zb + k (thread 0)
  auto refill = [&](int k) {
    uint64_t* bar = &bars[k % NS];
    mbar_arrive_expect_tx(bar, static_cast<uint32_t>(Sh::SLOT));
    tma_load_4d(slots + size_t(k % NS) * NC * NTM, tmap_p, x0, y0, zwrap(zb + k + NS), 0, bar);
    ++issued;
  };

  // gathered populations of three destination planes; the roles of the sets
  // are permuted at compile time
  R G[3][Q];
  produce(0, G[1][0], G[0][zm], G[2][zp]);
  window_ready(0);
  window_wait(0);

  // trip t, plane g = zb + 3 t + k
  auto sweep_plane = [&](const int t, auto K) {
    constexpr int k = decltype(K)::value;
    const int g = zb + 3 * t + k;
    const int kc = 3 * t + k + 1;  // plane c's index
    R(&G0)[Q] = G[k % 3];        // destination plane g - 1
    R(&G1)[Q] = G[(k + 1) % 3];  // g
    R(&G2)[Q] = G[(k + 2) % 3];  // g + 1
    const int c = g + 1;
    const R* win_g = win0 + k * WSTRIDE + wbase;
    R* win_c = win0 + ((k + 1) % 3) * WSTRIDE + wbase;
    R up_c = R(0);  // plane c's +z population: of plane c + 1, whose set is G0
    const R down_g = G0[zm], up_g = G2[zp];  // this node's own, for a z wall's bounce-back
    const bool z_lo = z_walls && g == 0, z_hi = z_walls && g == nz - 1;
    if (c <= ze) {
      produce(kc, G2[0], G1[zm], up_c);
      window_ready(kc);
    }

    if (active) {
      if (g <= ze) {
        static_for<1, Q>([&](auto A_) {
          constexpr int a = decltype(A_)::value;
          constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
          if constexpr (is_lateral<L>(a)) {
            const R v = win_g[lat_index<L>(a) * WPLANE - cy * WX - cx];
            if constexpr (cz == -1) G0[a] = v;
            if constexpr (cz == 0) G1[a] = v;
            if constexpr (cz == 1) G2[a] = v;
          }
        });
        // halfway bounce-back for destination plane g (threads next to a wall)
        if (xy_wall || z_lo || z_hi) {
          static_for<1, Q>([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            constexpr int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
            int cb = 0;
            if constexpr (cx == 1) cb |= bxlo ? 1 : 0;
            if constexpr (cx == -1) cb |= bxhi ? 1 : 0;
            if constexpr (cy == 1) cb |= bylo ? 2 : 0;
            if constexpr (cy == -1) cb |= byhi ? 2 : 0;
            if constexpr (cz == 1) cb |= z_lo ? 4 : 0;
            if constexpr (cz == -1) cb |= z_hi ? 4 : 0;
            if (cb != 0) {
              constexpr int oa = L::opp(a);
              R back;
              if constexpr (is_lateral<L>(oa)) back = win_g[lat_index<L>(oa) * WPLANE];
              else back = oa == zm ? down_g : up_g;
              const R v = back + args.bb[a][cb];
              // a descending link is gathered with plane c: its value waits in
              // the window cell it would be pulled from, which lies beyond the
              // wall and has no other writer or reader (beyond a z wall no
              // plane c is gathered)
              if constexpr (cz == -1 && is_lateral<L>(a)) {
                if (z_hi) G1[a] = v;
                else win_c[lat_index<L>(a) * WPLANE - cy * WX - cx] = v;
              } else {
                G1[a] = v;
              }
            }
          });
        }
      }
      // plane g - 1 is complete: collide it
      const int zd = g - 1;
      if (zd >= z0) {
        R fr[Q];
        static_for<0, Q>([&](auto A_) {
          constexpr int a = decltype(A_)::value;
          fr[a] = round_to_storage<S, R>(G0[a]);
        });
        Mom<R> m;
        moments<L, R, FORCE>(fr, args.ph, m);
        Coef<R> kc;
        coeffs<L, R, FORCE>(m, args.ph, kc);
        char* o = reinterpret_cast<char*>(out0 + plane * zd);
        const uint32_t v32 = args.vol32;
        each_coef<L, R>(kc, [&](auto I, R& v) {
          *reinterpret_cast<R*>(o + uint64_t(v32) * uint32_t(decltype(I)::value * 32 * sizeof(R))) = v;
        });
      }
    }
    G0[zp] = up_c;
    if (c <= ze) {
      window_wait(kc);
      // every thread has read plane c's slot
      if (tid == 0 && !dead && c + NS <= ze) refill(kc);
    }
  };
  // the slot of plane zb is free once its window is complete
  if (tid == 0 && !dead && zb + NS <= ze) refill(0);
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

template <class L, class S, class R, int BX, int BY, int NS, bool FORCE, int MINB>
__global__ void __launch_bounds__(K3Shape<L, R, BX, BY, NS, MINB>::NT, MINB)
    k3_step(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ K3Args<R> args) {
  const int b = blockIdx.x;
  k3_brick<L, S, R, BX, BY, NS, FORCE, MINB>(&tmap, args, b % args.ntx, (b / args.ntx) % args.nty,
                                             b / (args.ntx * args.nty));
}

// Populations -> coefficient fields, node by node (each thread reads all of
// its node's populations before it writes, so the fields may lie in the
// population array).
template <class L, class S, class R, bool FORCE>
__global__ void __launch_bounds__(256) k3_enter(const S* f, R* dst, int64_t vol, int nx, int pitch, Phys<R> ph) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < vol; i += int64_t(gridDim.x) * blockDim.x) {
    // rows are whole 32-element segments; the padding of a row stays zero
    const uint32_t seg = uint32_t(i >> 5) % uint32_t(pitch >> 5);
    if (int(seg * 32 + (i & 31)) >= nx) continue;
    R fr[L::Q];
    static_for<0, L::Q>([&](auto A_) {
      constexpr int a = decltype(A_)::value;
      fr[a] = load_as<S, R>(f[a * vol + i]);
    });
    Mom<R> m;
    moments<L, R, FORCE>(fr, ph, m);
    Coef<R> kc;
    coeffs<L, R, FORCE>(m, ph, kc);
    each_coef<L, R>(kc, [&](auto I, R& v) { dst[decltype(I)::value * vol + i] = v; });
  }
}

}  // namespace lbgb
