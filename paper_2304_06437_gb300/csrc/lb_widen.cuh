// lb_widen.cuh -- FP32 data to FP64 results without FP64 instructions.
//
// GB300 converts to and adds in FP64 at 1/64 of its FP32 rate (about 0.55 T
// operations a second in all), which bounds readouts of FP32 data long before
// the memory does.  The functions below give the values of the FP64
// instructions, bit for bit, from integer ones.
#pragma once

#include <cstdint>

#include "lb_collide.cuh"

namespace lbgb {

// double(v)
LB_DEV double widen(float v) {
  const uint32_t b = __float_as_uint(v), sign = b & 0x80000000u, m = b & 0x7fffffu, e = (b >> 23) & 0xffu;
  if (e == 0) {
    // a subnormal m 2^-149: its leading bit p is the implied one
    const int p = 31 - __clz(int(m));
    const uint64_t f = m ? uint64_t(p + 874) << 52 | (uint64_t(m) << (52 - p) & 0xfffffffffffffull) : 0;
    return __longlong_as_double(int64_t(uint64_t(sign) << 32 | f));
  }
  const uint32_t x = e == 0xffu ? 0x7ffu : e + 896;
  return __hiloint2double(int(sign | x << 20 | m >> 3), int(b << 29));
}
LB_DEV double widen(double v) { return v; }

// out = double(v) + c for a normal c > 0 of which cb are the bits: v in units of
// c's last place, rounded to nearest even, is added to the bits of c.  False for
// a sum that leaves c's binade or comes to its lower end (an exact sum below it
// has more places to keep): it takes the FP64 instructions, which the caller
// keeps out of the way (a predicated instruction that does nothing still takes
// its time in the FP64 pipe).
LB_DEV bool add_wide(float v, int64_t cb, double& out) {
  const int32_t b = __float_as_int(v);
  const int e = (b >> 23) & 0xff;
  const int m = (b & 0x7fffff) | (e ? 0x800000 : 0);
  const int sm = b < 0 ? -m : m;
  const int s = max(e, 1) + 925 - int(cb >> 52);  // v = sm 2^s units
  int64_t r = cb;
  if (s >= 0) {
    r += static_cast<int64_t>(sm) << min(s, 28);
  } else {
    const int k = min(-s, 30);
    const int q = sm >> k, rem = sm & ((1 << k) - 1), half = 1 << (k - 1);
    r += q;
    r += rem > half || (rem == half && (r & 1)) ? 1 : 0;
  }
  out = __longlong_as_double(r);
  return s <= 28 && e != 0xff && (r - 1) >> 52 == cb >> 52;
}
LB_DEV bool add_wide(double v, int64_t cb, double& out) {
  out = v + __longlong_as_double(cb);
  return true;
}

// t_a r for the lattice's |c|^2 shells, formed once on the host
struct ShellSums {
  double c[4];
};
template <class L>
ShellSums shell_sums(double r) {
  ShellSums s{};
  for (int a = 0; a < L::Q; ++a) s.c[L::shell(a)] = weight<L>(a) * r;
  return s;
}

// the shell of direction a in bits 2 a, 2 a + 1
template <class L>
LB_HD constexpr uint64_t shell_bits() {
  uint64_t m = 0;
  for (int a = 0; a < L::Q; ++a) m |= uint64_t(L::shell(a)) << (2 * a);
  return m;
}

// out[a n] = double(value of population a, p[a vol]) + t_a r
template <class L, class S, class R>
LB_DEV void widen_populations(const S* p, int64_t vol, double* out, int64_t n, const ShellSums& sums) {
  // every load before the first branch: all in flight together
  R v[L::Q];
#pragma unroll
  for (int a = 0; a < L::Q; ++a) v[a] = load_as<S, R>(p[a * vol]);
  uint32_t left = 0;
  static_for<0, L::Q>([&](auto A_) {
    constexpr int a = decltype(A_)::value;
    double r;
    if (!add_wide(v[a], __double_as_longlong(sums.c[L::shell(a)]), r)) left |= 1u << a;
    out[a * n] = r;
  });
  while (left) {
    const int a = __ffs(int(left)) - 1;
    left &= left - 1;
    constexpr uint64_t shells = shell_bits<L>();
    out[a * n] = static_cast<double>(load_as<S, R>(p[a * vol])) + sums.c[shells >> (2 * a) & 3];
  }
}

}  // namespace lbgb
