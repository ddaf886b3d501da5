// start.cu - FP32 states: initialisation from FP64 fields and conservation sums.
//
// Both are FP64 computations beside an FP32 state, and on the FP64 pipe that is
// what they took: 135 instructions a node for the equilibrium, 78 for the sums,
// 64 cycles each per SM sub-partition.  Here they run on the FP32 pipe with the
// errors carried along (dfloat.cuh); a node whose values leave the range that
// arithmetic is made for takes the FP64 formulas.  4096 x 1024 on GB300, the
// start of a run (mrtlb_init_equilibrium, mrtlb_reduce, mrtlb_get_f): 2.02 ->
// 0.53 ms, of which the sums' and the state's bytes alone are 0.18.
#include "dfloat.cuh"
#include "kernels.cuh"

namespace mrtlb {
namespace {

// The family inverses (Coef) as pairs of floats.
struct InverseDF {
  DF S[4][4], X[4][4], Y[4][4], Q[2][2], P[2][2];
};
DF host_df(double x) {
  const float h = (float)x;
  return DF{h, (float)(x - (double)h)};
}
InverseDF inverse_df(const Coef<double>& c) {
  InverseDF t;
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) {
      t.S[a][b] = host_df(c.invS[a][b]);
      t.X[a][b] = host_df(c.invX[a][b]);
      t.Y[a][b] = host_df(c.invY[a][b]);
    }
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      t.Q[a][b] = host_df(c.invQ[a][b]);
      t.P[a][b] = host_df(c.invP[a][b]);
    }
  return t;
}

// f = M^-1 f^eq(rho, u, T), versions 1 and 2 (Eqs. 14a-14i; see equilibrium()).
template <int VER>
__device__ __forceinline__ void equilibrium_df(const InverseDF& c, DF rho, DF ux, DF uy, DF T, float f[16]) {
  const DF x2 = df_mul(ux, ux), y2 = df_mul(uy, uy), xy = df_mul(ux, uy);
  const DF u2 = df_add(x2, y2), d2 = df_sub(x2, y2);
  const DF h = df_add(T, df_scale(u2, 0.5f));  // e / rho
  const DF e = df_mul(rho, h), jx = df_mul(rho, ux), jy = df_mul(rho, uy), k = df_mul(rho, u2);
  const DF ep = df_mul(rho, df_add(h, T));  // e + p
  const DF m4 = df_mul(rho, d2), m5 = df_mul(jx, uy), m6 = df_mul(ep, ux), m7 = df_mul(ep, uy);
  const DF m8 = df_mul(jx, df_sub(x2, df_mul(y2, 3.0f))), m9 = df_mul(jy, df_sub(df_mul(x2, 3.0f), y2));
  const DF m10 = df_sub(df_scale(df_mul(e, h), 2.0f), df_scale(df_mul(k, u2), 0.25f));
  const DF w = df_sub(df_mul(e, 6.0f), df_scale(k, 2.0f));
  const DF m12 = df_mul(w, d2), m13 = df_mul(w, xy);
  DF m14{0.0f, 0.0f}, m15{0.0f, 0.0f};
  if (VER == 2) {  // rho ux (5 d2 + (10 T - 4)), rho uy (5 d2 - (10 T - 4))
    const DF g = df_add(df_mul(T, 10.0f), DF{-4.0f, 0.0f}), q = df_mul(d2, 5.0f);
    m14 = df_mul(jx, df_add(q, g));
    m15 = df_mul(jy, df_sub(q, g));
  }
  constexpr int N = (VER == 2) ? 4 : 3;  // rows 14 and 15 are zero in version 1
  DF S[4], X[4], Y[4], Q[2], P[2];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    DF a = df_first(c.S[s][0], rho);  // (row 11 is zero in both)
    df_accumulate(a, c.S[s][1], e);
    df_accumulate(a, c.S[s][2], m10);
    S[s] = a;
    a = df_first(c.X[s][0], jx);
    df_accumulate(a, c.X[s][1], m6);
    df_accumulate(a, c.X[s][2], m8);
    if (N == 4) df_accumulate(a, c.X[s][3], m14);
    X[s] = a;
    a = df_first(c.Y[s][0], jy);
    df_accumulate(a, c.Y[s][1], m7);
    df_accumulate(a, c.Y[s][2], m9);
    if (N == 4) df_accumulate(a, c.Y[s][3], m15);
    Y[s] = a;
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    Q[s] = df_first(c.Q[s][0], m4);
    df_accumulate(Q[s], c.Q[s][1], m12);
    P[s] = df_first(c.P[s][0], m5);
    df_accumulate(P[s], c.P[s][1], m13);
  }
  auto put = [&](int q, DF a, DF b) {
    const DF v = df_join(a, b);
    f[q] = __fadd_rn(v.hi, v.lo);
  };
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s == 0 || s == 2) {
      const DF sp = df_join(S[s], Q[s >> 1]), sm = df_join(S[s], df_neg(Q[s >> 1]));
      put(4 * s + 0, sp, X[s]);
      put(4 * s + 2, sp, df_neg(X[s]));
      put(4 * s + 1, sm, Y[s]);
      put(4 * s + 3, sm, df_neg(Y[s]));
    } else {
      const DF sp = df_join(S[s], P[s >> 1]), sm = df_join(S[s], df_neg(P[s >> 1]));
      const DF a = df_join(X[s], Y[s]), b = df_join(X[s], df_neg(Y[s]));
      put(4 * s + 0, sp, a);
      put(4 * s + 2, sp, df_neg(a));
      put(4 * s + 1, sm, df_neg(b));
      put(4 * s + 3, sm, b);
    }
  }
}

// Whether equilibrium_df stays inside FP32's range: its largest terms are
// rho (u^2 + T)^2 times less than 2^13, in the fields' exponents 2^(r + 2 m + 13)
// with m the larger of T's and twice u's.  (Small terms may fall below the range:
// what they lose is 2^-149 beside f, which is of rho's size, 2^-60 or more.)
__device__ __forceinline__ int exponent(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }
__device__ __forceinline__ bool equilibrium_df_fits(double rho, double ux, double uy, double T) {
  const int m = max(exponent(T), 2 * max(exponent(ux), exponent(uy)));
  return df_fits(rho) && df_fits(ux) && df_fits(uy) && df_fits(T) && exponent(rho) + 2 * m <= 100;
}

template <int VER>
__global__ void __launch_bounds__(128) init_eq_df_kernel(const double* __restrict__ rho_in, const double* __restrict__ ux_in,
                                                         const double* __restrict__ uy_in, const double* __restrict__ T_in,
                                                         float* __restrict__ f, const Layout L,
                                                         const __grid_constant__ InverseDF c,
                                                         const __grid_constant__ Coef<double> c64) {
  const int i = blockIdx.y * 128 + threadIdx.x;
  const int j = blockIdx.x;
  if (i >= L.nx) return;
  const long long t = (long long)j * L.nx + i;
  const double rho = rho_in[t], ux = ux_in[t], uy = uy_in[t], T = T_in[t];
  float g[16];
  if (equilibrium_df_fits(rho, ux, uy, T)) {
    equilibrium_df<VER>(c, df_of(rho), df_of(ux), df_of(uy), df_of(T), g);
  } else {
    double eq[16], d[16];
    equilibrium<double, VER>(c64, rho, 1.0 / rho, rho * ux, rho * uy, rho * (T + 0.5 * (ux * ux + uy * uy)), ux, uy, T, eq);
    inverse_full(c64, eq, d);
#pragma unroll
    for (int q = 0; q < 16; ++q) g[q] = (float)d[q];
  }
  float* out = f + L.node(i, j);
#pragma unroll
  for (int q = 0; q < 16; ++q) out[q * L.plane] = g[q];
}

// rho, j_x, j_y, e of one node, each the sum of 16 floats times powers of two,
// rounded once (FP64 additions rounded at every step).
__device__ __forceinline__ void node_sums(const float g[16], F3& rho, F3& jx, F3& jy, F3& e) {
  rho = f3_of(g[0], g[1]);
  e = f3_of(0.5f * g[0], 0.5f * g[1]);
  jx = f3_of(g[0], -g[2]);
  jy = f3_of(g[1], -g[3]);
#pragma unroll
  for (int q = 2; q < 16; ++q) {
    const int vx = vx_of(q), vy = vy_of(q);
    f3_add(rho, g[q]);
    f3_add(e, 0.5f * (vx * vx + vy * vy) * g[q]);
    if (q > 2 && vx != 0) f3_add(jx, (float)vx * g[q]);
    if (q > 3 && vy != 0) f3_add(jy, (float)vy * g[q]);
  }
}

// (three blocks per SM, 80 registers: the same time as two or four)
constexpr int kSumThreads = 256, kSumBlocks = 3;
__global__ void __launch_bounds__(kSumThreads, kSumBlocks)
    reduce_f32_kernel(const float* __restrict__ f, double* acc, double* __restrict__ Tprev, int have_prev, const Layout L) {
  const long long stride = (long long)gridDim.x * kSumThreads, n = (long long)L.nx * L.ny;
  long long t = (long long)blockIdx.x * kSumThreads + threadIdx.x;
  const int dj = (int)(stride / L.nx), di = (int)(stride % L.nx);
  int i = (int)(t % L.nx), j = (int)(t / L.nx);
  F3 s[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k] = F3{0.0f, 0.0f, 0.0f};
  double out[4] = {0.0, 0.0, 0.0, 0.0}, mx = 0.0;
  for (; t < n; t += stride) {
    const float* at = f + L.node(i, j);
    float g[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) g[q] = at[q * L.plane];
    F3 m[4];
    node_sums(g, m[0], m[1], m[2], m[3]);
    double T;
    if (fabsf(m[0].a) + fabsf(m[3].a) < 1.152921504606847e18f && fabsf(m[0].a) > 8.673617379884035e-19f) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        f3_add(s[k], m[k].a);
        f3_add(s[k], m[k].b);
        if (m[k].c != 0.0f) f3_add(s[k], m[k].c);
      }
      const double rho = f3_value(m[0]), jx = f3_value(m[1]), jy = f3_value(m[2]), e = f3_value(m[3]);
      // 1 / rho from the FP32 reciprocal r by r (1 + d + d^2), d = 1 - rho r
      const double r = wide(recip(m[0].a)), d = fma(-rho, r, 1.0);
      T = temperature_plain(rho, jx, jy, e, fma(r, fma(d, d, d), r));
    } else {  // zero, subnormal, huge or not finite
      double v[16], rho, jx, jy, e;
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = (double)g[q];
      conserved(v, rho, jx, jy, e);
      out[0] += rho; out[1] += jx; out[2] += jy; out[3] += e;
      T = temperature_plain(rho, jx, jy, e, 1.0 / rho);
    }
    if (have_prev) {
      const double d = fabs(T - Tprev[t]);
      mx = (d > mx || d != d) ? d : mx;
    }
    Tprev[t] = T;
    i += di;
    j += dj;
    if (i >= L.nx) {
      i -= L.nx;
      ++j;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) out[k] += f3_value(s[k]);
  // one atomic per block and sum
  __shared__ double part[kSumThreads / 32][5];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] += __shfl_xor_sync(0xffffffffu, out[k], o);
    const double m = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = (m > mx || m != m) ? m : mx;
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) part[warp][k] = out[k];
    part[warp][4] = mx;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    const int k = threadIdx.x;
    double v = part[0][k];
    for (int w = 1; w < kSumThreads / 32; ++w) {
      const double p = part[w][k];
      v = (k < 4) ? v + p : (p > v || p != p) ? p : v;
    }
    // non-negative doubles order like their bit patterns; NaN maps above inf
    if (k < 4) {
      // the addition's own rounding, known from what was there, is summed beside
      // it: hundreds of blocks arriving in any order took 5 units in the last
      // place of a sum of 60,000 nodes
      const double old = atomicAdd(acc + k, v), s = old + v, b = s - old;
      const double e = (old - (s - b)) + (v - b);
      if (e != 0.0 && isfinite(e)) atomicAdd(acc + 5 + k, e);
    } else atomicMax((unsigned long long*)(acc + 4), (unsigned long long)__double_as_longlong(v));
  }
}

}  // namespace

bool launch_init_eq_df(const double* rho, const double* ux, const double* uy, const double* T, float* f, const Layout& L,
                       const Coef<double>& c64, cudaStream_t st) {
  if (c64.version > 2) return false;  // (the exponentials of version 3)
  const long long pieces = ((long long)L.nx + 127) / 128;
  if (pieces > 65535) return false;
  const dim3 grd(L.ny, (unsigned)pieces);
  const auto kernel = c64.version == 2 ? init_eq_df_kernel<2> : init_eq_df_kernel<1>;
  kernel<<<grd, 128, 0, st>>>(rho, ux, uy, T, f, L, inverse_df(c64), c64);
  return true;
}

void launch_reduce_f32(const float* f, double* acc, double* Tprev, int have_prev, const Layout& L, cudaStream_t st) {
  const long long n = (long long)L.nx * L.ny, blocks = (n + kSumThreads - 1) / kSumThreads, most = (long long)kSumBlocks * sm_count();
  reduce_f32_kernel<<<(unsigned)(blocks < most ? blocks : most), kSumThreads, 0, st>>>(f, acc, Tprev, have_prev, L);
}

}  // namespace mrtlb
