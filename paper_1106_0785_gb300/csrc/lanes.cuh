// lanes.cuh - a node on 16 lanes, one velocity each (step_split.cu says how).
#pragma once

#include "physics.cuh"

namespace mrtlb {
namespace {

constexpr unsigned kAll = 0xffffffffu;

template <typename R>
__device__ __forceinline__ R from_lane(R v, int l) { return __shfl_sync(kAll, v, l, 16); }
template <typename R>
__device__ __forceinline__ R across(R v, int m) { return __shfl_xor_sync(kAll, v, m, 16); }

// 1/x: FP32 as the other step kernels form it; FP64 by two Newton-Raphson steps
// r <- r + r (1 - x r) from the hardware's approximation, each squaring its
// relative error (four fused multiply-adds instead of the correctly rounded
// quotient's nine or so instructions; within one ulp of it).  Where the steps
// would leave the range (zeros, infinities, NaNs, magnitudes beyond 2^+-1021)
// the approximation stands: 1/0 = inf and 1/inf = 0 as the quotient has them.
__device__ __forceinline__ float split_recip(float x) { return recip(x); }
__device__ __forceinline__ double split_recip(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  double n = fma(r, fma(-x, r, 1.0), r);
  n = fma(n, fma(-x, n, 1.0), n);
  const unsigned e = (unsigned)__double2hiint(x) & 0x7ff00000u;
  return (e - (2u << 20) <= (2042u << 20)) ? n : r;  // biased exponents 2 .. 2044
}

// The lane's constants that follow from its place.
template <typename R>
struct Lane {
  int l, s, k;
  bool axis, half;  // axis: shells of axis velocities; half: an axis shell's X or Y
  __device__ __forceinline__ explicit Lane(int lane) : l(lane & 15), s((lane & 15) >> 2), k(lane & 3) {
    axis = (s & 1) == 0;
    half = axis && k >= 2;
  }
  // f_l -> harmonic k of shell s
  __device__ __forceinline__ R harmonic(R v) const {
    R o = across(v, 2);
    v = (k < 2) ? v + o : o - v;
    o = across(v, 1);
    if (!axis && k == 2) o = -o;
    return v * (k == 1 ? R(-1) : R(1)) + (half ? R(0) : o);
  }
  // harmonic k of shell s -> the value at velocity l (pre-scaled harmonics)
  __device__ __forceinline__ R velocity(R v) const {
    R o = across(v, 1);
    v = v * ((k == 1 || (k == 3 && !axis)) ? R(-1) : R(1)) + (half ? R(0) : o);
    o = across(v, 2);
    if (k == 1 && !axis) o = -o;
    return v * ((k == 2 || (k == 3 && axis)) ? R(-1) : R(1)) + o;
  }
  // m - m^eq of the lane's moment (halves of moments 10, 12 and 13), version 1;
  // m itself where the equilibrium is the moment or zero.  t = rho |u|^2.
  __device__ __forceinline__ R departure(R m, R rho, R ir, R jx, R jy, R e, R ux, R uy, R t, R p) const {
    const bool is10 = l == 8, is12 = l == 9, is13 = l == 13, is9 = l == 11;
    const R z1 = (is10 ? e : ux) * (is10 ? e : is13 ? uy : ux);
    const R q2 = is10 ? t : uy;
    const R z2 = q2 * q2;
    R z = (is9 ? R(3) : is10 ? R(-0.125) : l == 10 ? R(-3) : is13 ? R(0) : R(-1)) * (is9 ? z1 : z2) + (is9 ? -z2 : z1);
    if (l == 5 || l == 7) z = uy;  // m5, m7
    if (l == 6) z = ux;            // m6
    const bool is67 = l == 6 || l == 7;
    const R aw = (is67 ? R(1) : R(3)) * e + (is67 ? p : -t);
    R a = R(0);
    if (l == 1) a = rho;               // m4 = rho (ux^2 - uy^2)
    if (l == 5 || l == 10) a = jx;     // m5 = jx uy, m8 = jx (ux^2 - 3 uy^2)
    if (l == 11) a = jy;               // m9 = jy (3 ux^2 - uy^2)
    if (is10) a = ir;                  // m10 / 2 = (e^2 - (rho u^2)^2 / 8) / rho
    if (is67 || is12 || is13) a = aw;  // (e + p) u; m12 / 2, m13 / 2: w / 2 = 3 e - rho u^2
    return m - a * z;
  }
  // moment s of family k from harmonic k of the four shells
  __device__ __forceinline__ R moment(R h, const R c[4]) const {
    R m = c[0] * from_lane(h, k);
#pragma unroll
    for (int r = 1; r < 4; ++r) m += c[r] * from_lane(h, 4 * r + k);
    return m;
  }
};

}  // namespace
}  // namespace mrtlb
