// lb_pair.cuh -- two FP32 lanes in one register pair, computed with the
// packed FP32x2 instructions of sm_100 and later (one issue slot for two
// node updates).
//
// Every operator is the lane-wise IEEE operation with round-to-nearest-even,
// exactly as the scalar FP32 instruction it replaces (a - b is evaluated as
// a + (-b), which rounds identically), so the per-node arithmetic of
// lb_collide.cuh instantiated with f32x2 produces, lane by lane, the same bits
// as its scalar float instantiation.
#pragma once

#include "lb_collide.cuh"

namespace lbgb {

struct f32x2 {
  float x, y;
  __host__ __device__ constexpr f32x2() : x(0.0f), y(0.0f) {}
  __host__ __device__ constexpr f32x2(float a, float b) : x(a), y(b) {}
  // broadcast (the scalar conversion of the value, in both lanes)
  __host__ __device__ constexpr explicit f32x2(float v) : x(v), y(v) {}
  __host__ __device__ constexpr explicit f32x2(double v) : x(float(v)), y(float(v)) {}
  __host__ __device__ constexpr explicit f32x2(int v) : x(float(v)), y(float(v)) {}
};

__device__ __forceinline__ float2 as_f2(f32x2 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ f32x2 of_f2(float2 v) { return f32x2(v.x, v.y); }

__device__ __forceinline__ f32x2 operator+(f32x2 a, f32x2 b) { return of_f2(__fadd2_rn(as_f2(a), as_f2(b))); }
__device__ __forceinline__ f32x2 operator-(f32x2 a) { return f32x2(-a.x, -a.y); }
__device__ __forceinline__ f32x2 operator-(f32x2 a, f32x2 b) { return of_f2(__fadd2_rn(as_f2(a), as_f2(-b))); }
__device__ __forceinline__ f32x2 operator*(f32x2 a, f32x2 b) { return of_f2(__fmul2_rn(as_f2(a), as_f2(b))); }
__device__ __forceinline__ f32x2 fma_r(f32x2 a, f32x2 b, f32x2 c) {
  return of_f2(__ffma2_rn(as_f2(a), as_f2(b), as_f2(c)));
}

// ------------------------------------------------------------ storage pairs
// two adjacent stored values <-> one f32x2 (the address must be aligned to
// two elements)
template <class S>
__device__ __forceinline__ f32x2 load_pair(const S* p);
template <>
__device__ __forceinline__ f32x2 load_pair<float>(const float* p) {
  return of_f2(*reinterpret_cast<const float2*>(p));
}
template <>
__device__ __forceinline__ f32x2 load_pair<__half>(const __half* p) {
  return of_f2(__half22float2(*reinterpret_cast<const __half2*>(p)));
}
template <>
__device__ __forceinline__ f32x2 load_pair<__nv_bfloat16>(const __nv_bfloat16* p) {
  return of_f2(__bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p)));
}

template <class S>
__device__ __forceinline__ void store_pair(S* p, f32x2 v);
template <>
__device__ __forceinline__ void store_pair<float>(float* p, f32x2 v) {
  *reinterpret_cast<float2*>(p) = as_f2(v);
}
template <>
__device__ __forceinline__ void store_pair<__half>(__half* p, f32x2 v) {
  // lane-wise round-to-nearest-even, as __float2half_rn
  *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v.x, v.y);
}
template <>
__device__ __forceinline__ void store_pair<__nv_bfloat16>(__nv_bfloat16* p, f32x2 v) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
}

template <class S>
__device__ __forceinline__ f32x2 round_pair(f32x2 v) {
  return f32x2(round_to_storage<S, float>(v.x), round_to_storage<S, float>(v.y));
}

// ---------------------------------------------------------- packed collision
// moments, coefficients and post-collision set of lb_collide.cuh for a pair of
// nodes, with every negation folded into a packed multiply-add or a negated
// constant (a packed operand has no sign modifier, so each would cost
// instructions of its own).  The values are those of the scalar functions
// (x - y and (-1) y + x round alike; negation is exact); only the sign of a
// zero can differ.
LB_DEV f32x2 sub_r(f32x2 a, f32x2 b) { return fma_r(b, f32x2(-1.0f), a); }

// the balanced sum of sign(k) * term(k): the value and, at compile time, the
// sign it carries (that of the first term)
template <int Lo, int Hi, class F, class G>
LB_DEV f32x2 signed_tree(F&& term, G sign) {
  if constexpr (Hi - Lo == 1) {
    return term(std::integral_constant<int, Lo>{});
  } else {
    constexpr int Mid = Lo + (Hi - Lo) / 2;
    const f32x2 a = signed_tree<Lo, Mid>(term, sign), b = signed_tree<Mid, Hi>(term, sign);
    if constexpr (G::of(Lo) == G::of(Mid)) return a + b;
    else return sub_r(a, b);
  }
}
template <class L, int al>
struct AxisSign {
  LB_HD static constexpr int of(int k) { return comp<L>(al, pair_first<L>(axis_pair<L>(al, k))); }
};
template <class L, int al, int be>
struct OdSign {
  LB_HD static constexpr int of(int k) {
    return comp<L>(al, pair_first<L>(od_pair<L>(al, be, k))) * comp<L>(be, pair_first<L>(od_pair<L>(al, be, k)));
  }
};

template <class L, bool FORCE>
LB_DEV void moments_coeffs(const f32x2 (&f)[L::Q], const Phys<f32x2>& ph, Coef<f32x2>& kc) {
  using V = f32x2;
  constexpr int NP = n_pairs<L>();
  V s[NP], t[NP];
  static_for<0, NP>([&](auto P) {
    constexpr int p = decltype(P)::value;
    constexpr int a = pair_first<L>(p);
    s[p] = f[a] + f[L::opp(a)];
    t[p] = sub_r(f[a], f[L::opp(a)]);
  });
  const V drho = tree_sum<0, NP + 1, V>([&](auto K) -> V {
    constexpr int k = decltype(K)::value;
    if constexpr (k == 0) return f[0];
    else return s[k - 1];
  });
  V u[3] = {V(0), V(0), V(0)}, nru[3] = {V(0), V(0), V(0)}, pi[6] = {V(0), V(0), V(0), V(0), V(0), V(0)};
  static_for<0, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    if constexpr (L::axis(al)) {
      constexpr int n = axis_pair_count<L>(al);
      const V j = signed_tree<0, n>([&](auto K) -> V { return t[axis_pair<L>(al, decltype(K)::value)]; },
                                    AxisSign<L, al>{});
      constexpr bool pos = AxisSign<L, al>::of(0) == 1;
      if constexpr (FORCE) u[al] = (pos ? j + ph.hF[al] : sub_r(ph.hF[al], j)) * ph.inv_rho0;
      else u[al] = j * (pos ? ph.inv_rho0 : ph.n_inv_rho0);
      nru[al] = ph.n_rho0 * u[al];
    }
  });
  static_for<0, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    if constexpr (L::axis(al)) {
      constexpr int n = axis_pair_count<L>(al);
      const V Pd = tree_sum<0, n, V>([&](auto K) -> V { return s[axis_pair<L>(al, decltype(K)::value)]; });
      pi[al] = fma_r(nru[al], u[al], fma_r(ph.n_cs2, drho, Pd));
      static_for<al + 1, 3>([&](auto BE) {
        constexpr int be = decltype(BE)::value;
        if constexpr (L::axis(be)) {
          constexpr int no = od_pair_count<L>(al, be);
          const V Po = signed_tree<0, no>([&](auto K) -> V { return s[od_pair<L>(al, be, decltype(K)::value)]; },
                                          OdSign<L, al, be>{});
          // (negative leading sign: -Po - rho0 u u, as (-1) Po + nru u)
          if constexpr (OdSign<L, al, be>::of(0) == 1) pi[3 + od(al, be)] = fma_r(nru[al], u[be], Po);
          else pi[3 + od(al, be)] = fma_r(nru[al], u[be], Po * V(-1.0f));
        }
      });
    }
  });
  V usq = u[0] * u[0], tr = pi[0], uF = u[0] * ph.F[0];
  static_for<1, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    if constexpr (L::axis(al)) {
      usq = fma_r(u[al], u[al], usq);
      tr = tr + pi[al];
      if constexpr (FORCE) uF = fma_r(u[al], ph.F[al], uF);
    }
  });
  kc.A = fma_r(ph.n15om1, tr, fma_r(ph.n15rho0, usq, drho));
  if constexpr (FORCE) kc.A = fma_r(ph.n3g, uF, kc.A);
  static_for<0, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    if constexpr (L::axis(al)) {
      V b = ph.c3rho0 * u[al];
      V c = fma_r(ph.c45om1, pi[al], (ph.c45rho0 * u[al]) * u[al]);
      if constexpr (FORCE) {
        b = fma_r(V(1.5f), ph.F[al], b);
        c = fma_r(ph.c9g, u[al] * ph.F[al], c);
      }
      kc.B[al] = b;
      kc.C[al] = c;
      static_for<al + 1, 3>([&](auto BE) {
        constexpr int be = decltype(BE)::value;
        if constexpr (L::axis(be)) {
          V o = fma_r(ph.c9om1, pi[3 + od(al, be)], (ph.c9rho0 * u[al]) * u[be]);
          if constexpr (FORCE) o = fma_r(ph.c9g, fma_r(u[al], ph.F[be], ph.F[al] * u[be]), o);
          kc.C2[od(al, be)] = o;
        }
      });
    }
  });
}

// even part and unscaled odd part of direction a, whose first non-zero
// component is +1
template <class L, int a>
LB_DEV void post_even_odd(const Coef<f32x2>& k, f32x2& even, f32x2& odd) {
  even = k.A;
  static_for<0, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    if constexpr (comp<L>(al, a) != 0) even = even + k.C[al];
  });
  bool first = true;
  static_for<0, 3>([&](auto AL) {
    constexpr int al = decltype(AL)::value;
    constexpr int ca = comp<L>(al, a);
    static_for<al + 1, 3>([&](auto BE) {
      constexpr int be = decltype(BE)::value;
      constexpr int cc = ca * comp<L>(be, a);
      if constexpr (cc == 1) even = even + k.C2[od(al, be)];
      if constexpr (cc == -1) even = sub_r(even, k.C2[od(al, be)]);
    });
    if constexpr (ca != 0) {
      if (first) odd = k.B[al];
      else odd = ca == 1 ? odd + k.B[al] : sub_r(odd, k.B[al]);
      first = false;
    }
  });
}
template <class L>
LB_HD constexpr int leading_sign(int a) {
  return L::cx(a) != 0 ? L::cx(a) : (L::cy(a) != 0 ? L::cy(a) : L::cz(a));
}
// one population, and both members of a pair {a, opp(a)}, leading_sign(a) = 1
template <class L, int a>
LB_DEV f32x2 post_v(const Coef<f32x2>& k) {
  constexpr float w = float(weight<L>(a));
  if constexpr (a == 0) {
    return f32x2(w) * k.A;
  } else {
    constexpr int s = leading_sign<L>(a);
    f32x2 even, odd;
    post_even_odd<L, s == 1 ? a : L::opp(a)>(k, even, odd);
    return fma_r(f32x2(w), even, f32x2(s == 1 ? w : -w) * odd);
  }
}
template <class L, int a>
LB_DEV void post_pair(const Coef<f32x2>& k, f32x2& fa, f32x2& fo) {
  constexpr float w = float(weight<L>(a));
  f32x2 even, odd;
  post_even_odd<L, a>(k, even, odd);
  fa = fma_r(f32x2(w), even, f32x2(w) * odd);
  fo = fma_r(f32x2(w), even, f32x2(-w) * odd);
}

// the same names for the scalar types
template <class L, bool FORCE, class R>
LB_DEV void moments_coeffs(const R (&f)[L::Q], const Phys<R>& ph, Coef<R>& kc) {
  Mom<R> m;
  moments<L, R, FORCE>(f, ph, m);
  coeffs<L, R, FORCE>(m, ph, kc);
}
template <class L, int a, class R>
LB_DEV R post_v(const Coef<R>& k) {
  return post<L, R, a>(k);
}
template <class L, int a, class R>
LB_DEV void post_pair(const Coef<R>& k, R& fa, R& fo) {
  constexpr R w = R(weight<L>(a));
  R even, wodd;
  post_parts<L, R, a>(k, even, wodd);
  fa = fma_r(w, even, wodd);
  fo = fma_r(w, even, -wodd);
}

}  // namespace lbgb
