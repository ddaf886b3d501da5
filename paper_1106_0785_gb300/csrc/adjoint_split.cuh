// adjoint_split.cuh - the adjoint step of small grids: 16 lanes per node.
//
// As step_split.cu: a small grid's step takes as long as one thread's chain,
// in FP64 64 cycles an instruction.  The two-pass kernels spend 122 + 870 FP64
// instructions a node (4 x 200, version 1, with the rate gradients: 27 us for
// the second pass alone); one velocity and one moment per lane takes about 145
// for two nodes, in one launch:
//   * rho, e, j and the two modification moments of lambda at the four
//     neighbours by transposed sums, lane (s, k) ending with value k of
//     neighbour s; each group of four lanes then has its neighbour's u, and
//     the strain adjoints gbar of it;
//   * the equilibrium's transpose as a row of the Jacobian per lane, the
//     derivatives of its own moment by (rho, e, j_x, j_y), each a product of a
//     lane-chosen factor with a two-term sum (LaneJacobian), summed over the
//     lanes with the moments' adjoints;
//   * M^T back as the forward step's M^-1: moments to shells, two butterflies.
// Version 1; the other versions keep the kernels of larger grids.
#pragma once

#include "adjoint.cuh"
#include "lanes.cuh"

namespace mrtlb {
namespace {

template <typename R>
struct AdjSplitTable {
  R mom[4][16], inv_t[4][16], back[4][16];  // moment from harmonics, its adjoint from lambda's, harmonics from adjoints
  R rate[16], twice[16];                     // (2 where the lane holds half a moment)
  R wg[16], wl[16];                          // the shell's weight in the neighbours' moments of f, of lambda
  R dr[2][16], dx[2][16], dy[2][16], de[16]; // LaneJacobian
  R lw[4][16], selfw[16];
  R ga[16], gb[16];                          // rate gradients through the modification factors
};

// The derivatives of the lane's equilibrium moment (of moment 10, 12, 13
// itself, not its half) by rho, e, j_x, j_y: the weights are in the table.
template <typename R>
struct LaneJacobian {
  R rho, e, jx, jy;
  template <typename T>
  __device__ __forceinline__ LaneJacobian(const Lane<R>& me, const T& w, R ux, R uy, R h) {  // h = e / rho
    const int l = me.l;
    const R x2 = ux * ux, y2 = uy * uy, xy = ux * uy, u2 = x2 + y2, d2 = x2 - y2;
    const R W = R(3) * h - u2, E = R(2) * h - R(0.5) * u2;  // (3 e - rho u^2) / rho, (e + p) / rho
    const bool is12 = l == 9, is13 = l == 13, is10 = l == 8, is6 = l == 6, is7 = l == 7;
    const bool one = l == 1 || l == 5;
    const R y = w.dr[0] * (one ? R(1) : is10 ? h : (l == 10 || l == 11) ? x2 : u2) +
                w.dr[1] * ((is6 || is7) ? E : (is12 || is13) ? W : y2);
    rho = ((l == 1 || is12) ? d2 : (l == 5 || is13) ? xy : is10 ? h : (is7 || l == 11) ? uy : ux) * y;
    const R r10 = R(0.75) * u2;
    if (is10) rho = r10 * u2 + rho;
    const R ax = (is12 || is13) ? W : is10 ? u2 : is6 ? E : R(1), ay = (is12 || is13) ? W : is10 ? u2 : is7 ? E : R(1);
    jx = ((l == 1 || is10 || is12) ? ux : (l == 5 || is13) ? uy : is6 ? R(1) : l == 10 ? d2 : xy) *
         (w.dx[0] * ax + w.dx[1] * (is12 ? d2 : x2));
    jy = ((l == 1 || is10 || is12) ? uy : (l == 5 || is13) ? ux : is7 ? R(1) : l == 11 ? d2 : xy) *
         (w.dy[0] * ay + w.dy[1] * (is12 ? d2 : y2));
    e = w.de * (is6 ? ux : is7 ? uy : is10 ? h : is12 ? d2 : xy);
  }
};
// Sums over the 16 lanes of four values; lane k of each shell gets number k.
template <typename R>
__device__ __forceinline__ R sum_of_four(const Lane<R>& me, R a, R b, R c, R d) {
  const bool up = me.k >= 2, odd = me.k & 1;
  const R p = (up ? c : a) + across(up ? a : c, 2), q = (up ? d : b) + across(up ? b : d, 2);
  R v = (odd ? q : p) + across(odd ? p : q, 1);
  v += across(v, 4);
  return v + across(v, 8);
}
template <typename R>
struct JacobianWeights {
  R dr[2], dx[2], dy[2], de;
  __device__ __forceinline__ JacobianWeights(const AdjSplitTable<R>* t, int l) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      dr[q] = t->dr[q][l];
      dx[q] = t->dx[q][l];
      dy[q] = t->dy[q][l];
    }
    de = t->de[l];
  }
};

constexpr int kAdjSplitThreads = 64;

// lambda~ of every node of [-1, nx] x [-1, ny] but the corners.
template <typename R, bool RATES>
__global__ void __launch_bounds__(kAdjSplitThreads)
    adj_split_kernel(const R* __restrict__ ft, const R* __restrict__ lam, R* __restrict__ out, const Layout L,
                     const AdjSplitTable<R>* __restrict__ tab, const R mod0, const R mod1, const R mod2, const R mod3,
                     const R inv2dx, const R inv2dy, const int modified, double* gacc) {
  const Lane<R> me(threadIdx.x);
  const int l = me.l, s = me.s, k = me.k;
  const int nx2 = L.nx + 2, n = nx2 * (L.ny + 2);
  const int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  const int t0 = min(id, n - 1);
  const int i = t0 % nx2 - 1, j = t0 / nx2 - 1;
  const bool live = id < n && !((i < 0 || i >= L.nx) && (j < 0 || j >= L.ny));
  const bool adv = live && advanced<R>(L, i, j);
  R cm[4], ct[4], cb_[4], lw[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    cm[r] = tab->mom[r][l];
    ct[r] = tab->inv_t[r][l];
    cb_[r] = tab->back[r][l];
    lw[r] = tab->lw[r][l];
  }
  const JacobianWeights<R> jw(tab, l);
  const R rate = tab->rate[l], wg = tab->wg[l], wl = tab->wl[l], selfw = tab->selfw[l];
  after_previous();

  // neighbours E, W, N, S: in the padded grid, advanced, offset
  const bool in[4] = {i < L.nx, i >= 0, j < L.ny, j >= 0};
  const bool an[4] = {live && advanced<R>(L, i + 1, j), live && advanced<R>(L, i - 1, j), live && advanced<R>(L, i, j + 1),
                      live && advanced<R>(L, i, j - 1)};
  const long long off[4] = {1, -1, L.pitch, -(long long)L.pitch};
  const long long at = l * L.plane + L.node(i, j);
  const R f = ft[at], lo = lam[at];
  R fn[4], ln[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long a = at + (in[q] ? off[q] : 0);
    fn[q] = ft[a];
    ln[q] = lam[a];
  }
  const R lp = adv ? lo : R(0);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (!an[q]) ln[q] = R(0);

  // neighbour s: k = 0 rho, 1 e, 2 j_x, 3 j_y in vg; 2, 3: moments 6, 7 of -lambda in vl
  auto gather = [&](const R v[4], R w) {
    R h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      R o = across(v[q], 2);
      R x = (k < 2) ? v[q] + o : o - v[q];
      o = across(x, 1);
      if (!me.axis && k == 2) o = -o;
      h[q] = w * (x + ((me.half) ? R(0) : o));
    }
    const bool odd = s & 1, high = s >> 1;
    const R a = (odd ? h[1] : h[0]) + across(odd ? h[0] : h[1], 4);
    const R b = (odd ? h[3] : h[2]) + across(odd ? h[2] : h[3], 4);
    return (high ? b : a) + across(high ? a : b, 8);
  };
  const R vg = gather(fn, wg);
  const R m = me.moment(me.harmonic(f), cm);
  const R rho = from_lane(m, 0), e = from_lane(m, 4), jx = from_lane(m, 2), jy = from_lane(m, 3);
  const R rn = from_lane(vg, 4 * s), en = from_lane(vg, 4 * s + 1), jxn = from_lane(vg, 4 * s + 2), jyn = from_lane(vg, 4 * s + 3);
  // one reciprocal for the node (lanes k = 1) and its neighbours; cells without
  // an advanced node beside them (behind walls, beyond the padded grid) hold anything
  const R den = (k == 1) ? rho : rn;
  const R rec = (den > R(0)) ? split_recip(den) : R(0);
  const R ir = from_lane(rec, 1), irn = from_lane(rec, 4 * s);
  const R ux = jx * ir, uy = jy * ir;
  const R p = e - R(0.5) * (jx * ux + jy * uy);
  R uxb = R(0), uyb = R(0), shear = R(0), strain = R(0);
  if (modified) {
    const R vl = gather(ln, wl);
    const R c6 = -from_lane(vl, 4 * s + 2), c7 = -from_lane(vl, 4 * s + 3);
    const R uxn = jxn * irn, uyn = jyn * irn;
    const bool ev = (k & 1) == 0;
    const R pn = en - R(0.5) * (jxn * uxn + jyn * uyn);
    // even lanes: gbar_shear of neighbour s, odd ones gbar_strain
    const bool ans = s == 0 ? an[0] : s == 1 ? an[1] : s == 2 ? an[2] : an[3];
    R gb = pn * (c6 * ((ev ? mod0 : mod1) * (ev ? uxn : uyn)) + c7 * ((ev ? mod3 : mod2) * (ev ? uyn : uxn)));
    if (!ans) gb = R(0);
    const R dg = across(gb, 4) - gb;  // shells 0, 1: W - E; 2, 3: S - N (the odd shells: the negative)
    const R gx = from_lane(dg, ev ? 0 : 1), gy = from_lane(dg, ev ? 9 : 8);
    const R ub = gx * inv2dx + (ev ? gy * inv2dy : -(gy * inv2dy));
    uxb = from_lane(ub, 0);
    uyb = from_lane(ub, 1);
    // even lanes: shear of u at the node, odd ones strain
    const R du = (k < 2) ? uxn : uyn, dd = du - across(du, 4);  // E - W, N - S of u_x (k < 2) and u_y
    const R sx = from_lane(dd, ev ? 0 : 2), sy = from_lane(dd, ev ? 10 : 8);
    const R st = sx * inv2dx + (ev ? -(sy * inv2dy) : sy * inv2dy);
    shear = from_lane(st, 0);
    strain = from_lane(st, 1);
    if (!adv) shear = strain = R(0);
  }

  // the moments' adjoints -dC^T lambda, and the equilibrium's part of them
  const R cb = -me.moment(me.harmonic(lp), ct);
  const R mb = rate * cb;  // (zero at the conserved moments)
  const LaneJacobian<R> J(me, jw, ux, uy, e * ir);
  R acc = -sum_of_four<R>(me, mb * J.rho, mb * J.e, mb * J.jx, mb * J.jy);  // lane k: rho, e, j_x, j_y
  // the modification's own factors and everything through u
  const R c6 = from_lane(cb, 6), c7 = from_lane(cb, 7);
  R pb = R(0), gux = uxb, guy = uyb;
  if (modified) {
    const R gx = (c6 * mod0) * shear + (c7 * mod2) * strain, gy = (c6 * mod1) * strain + (c7 * mod3) * shear;
    pb = ux * gx + uy * gy;
    gux += p * gx;
    guy += p * gy;
  }
  const R u2h = R(0.5) * (ux * ux + uy * uy), gw = ux * gux + uy * guy;
  acc += (k == 0 ? -ir : k == 1 ? R(0) : ir) * (k == 0 ? gw : k == 2 ? gux : guy) +
         (k == 0 ? u2h : k == 1 ? R(1) : k == 2 ? -ux : -uy) * pb;
  // lanes of the conserved moments: rho (0, 0), e (1, 0), j_x (0, 2), j_y (0, 3)
  const R acc_e = from_lane(acc, 1);
  const R mbar = (l == 4) ? acc_e : (l == 0 || l == 2 || l == 3) ? acc : mb;
  const R local = me.velocity(me.moment(mbar, cb_));
  R lt = (adv || an[0] || an[1] || an[2] || an[3]) ? local : R(0);  // (else B(f) means nothing there: velocity_T)
  lt += selfw * lp;
  lt += lw[1] * ln[0];
  lt += lw[0] * ln[1];
  lt += lw[3] * ln[2];
  lt += lw[2] * ln[3];
  if (live) out[at] = lt;

  if constexpr (RATES) {
    const R t = jx * ux + jy * uy;
    R G = cb * (tab->twice[l] * me.departure(m, rho, ir, jx, jy, e, ux, uy, t, p));
    if (modified) {
      // s7, s8 (lanes 6, 7) and s5, s6 (lanes 1, 5) in the factors of the modification
      const bool second = l == 7 || l == 5;
      const R qa = p * (l == 5 ? uy : ux) * (second ? strain : shear);          // A0, A2, A0, A1
      const R qb = p * (l == 5 ? ux : uy) * ((l == 6 || l == 5) ? strain : shear);  // A1, A3, A3, A2
      G += (l == 7 ? c7 : c6) * qa * tab->ga[l] + (l == 6 ? c6 : c7) * qb * tab->gb[l];
    }
    if (!adv) G = R(0);
    __shared__ double part[kAdjSplitThreads / 32][16];
    G += __shfl_xor_sync(kAll, G, 16);
    if ((threadIdx.x & 31) < 16) part[threadIdx.x >> 5][l] = (double)G;
    __syncthreads();
    if (threadIdx.x < 16) {
      double sum = 0.0;
#pragma unroll
      for (int w = 0; w < kAdjSplitThreads / 32; ++w) sum += part[w][l];
      // the lane's moment: rows of (k = 0, 1, 2, 3)
      const int at4 = (k == 0) ? (s == 0 ? 0 : s == 1 ? 3 : 8 + s) : (k == 1) ? (s == 0 ? 4 : s == 1 ? 5 : 10 + s)
                    : (k == 2) ? (s == 0 ? 1 : s == 1 ? 6 : s == 2 ? 8 : 14) : (s == 0 ? 2 : s == 1 ? 7 : s == 2 ? 9 : 15);
      if (at4 >= 4 && sum != 0.0) atomicAdd(gacc + 16 * (blockIdx.x % kGradSlots) + at4, sum);
    }
  }
}

// adj_walls_kernel on 16 lanes per wall node (FP64 whatever the state's precision).
template <typename R>
__global__ void __launch_bounds__(32)
    adj_walls_split_kernel(R* lam, const R* __restrict__ ft, const Layout L, const AdjSplitTable<double>* __restrict__ tab,
                           const __grid_constant__ Walls w, const int side0, const int total) {
  const Lane<double> me(threadIdx.x);
  const int l = me.l;
  const int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  double cm[4], cf[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    cm[r] = tab->mom[r][l];
    cf[r] = tab->inv_t[r][l];
  }
  const JacobianWeights<double> jw(tab, l);
  const int n = (side0 < 2) ? L.ny : L.nx;
  const int kk = min(id, total - 1);
  const int side = side0 + (kk >= n), q = kk >= n ? kk - n : kk;
  const double ew = w.e64[side][l];
  after_previous();
  const int i = (side == 0) ? 0 : (side == 1) ? L.nx - 1 : q, j = (side == 2) ? 0 : (side == 3) ? L.ny - 1 : q;
  const long long aw = l * L.plane + L.node(i, j);
  const long long aa = aw + (side == 0 ? 1 : side == 1 ? -1 : side == 2 ? L.pitch : -(long long)L.pitch);
  const double v = (double)lam[aw], g = (double)ft[aa], la = (double)lam[aa];
  const double m = me.moment(me.harmonic(g), cm);
  const double rho = from_lane(m, 0), e = from_lane(m, 4), jx = from_lane(m, 2), jy = from_lane(m, 3);
  const double ir = split_recip(rho), ux = jx * ir, uy = jy * ir;
  // the equilibrium moments' adjoints: -M^-T lambda (the conserved ones too)
  const double eqb = -me.moment(me.harmonic(v), cf);
  const bool cons = l == 0 || (l >= 2 && l <= 4);
  const LaneJacobian<double> J(me, jw, ux, uy, e * ir);
  const double rw = v * ew;  // the wall state's equilibrium is rho times a constant
  // (the conserved moments' equilibria are themselves)
  const double r0 = ((l == 0) ? eqb : cons ? 0.0 : eqb * J.rho) + rw;
  const double e0 = (l == 4) ? eqb : cons ? 0.0 : eqb * J.e;
  const double x0 = (l == 2) ? eqb : cons ? 0.0 : eqb * J.jx;
  const double y0 = (l == 3) ? eqb : cons ? 0.0 : eqb * J.jy;
  const double s4 = sum_of_four<double>(me, r0, e0, x0, y0);
  const double rb = from_lane(s4, 0), eb = from_lane(s4, 1), jxb = from_lane(s4, 2), jyb = from_lane(s4, 3);
  const double vx = vx_of(l), vy = vy_of(l);
  const double add = v + rb + jxb * vx + jyb * vy + eb * (0.5 * (vx * vx + vy * vy));
  if (id < total) {
    lam[aa] = (R)(la + add);
    lam[aw] = R(0);
  }
}

template <typename R>
void adj_split_table(const AdjCoef<R>& a, const Coef<double>& c64, AdjSplitTable<R>* t) {
  static const double S[4][4] = {{1, 1, 1, 1}, {0.5, 1, 2, 4}, {0.25, 1, 4, 16}, {1, -4, 16, -64}};
  static const double X[4][4] = {{1, 1, 2, 2}, {0.5, 1, 4, 8}, {1, -2, 8, -16}, {1, -4, 32, -128}};
  static const double Q[4][4] = {{1, 0, 4, 0}, {0, 1, 0, 4}, {1, 0, 16, 0}, {0, 2, 0, 32}};
  static const int moment[4][4] = {{0, 4, 1, 2}, {3, 5, 6, 7}, {10, 12, 8, 9}, {11, 13, 14, 15}};  // [s][k]
  const Coef<double>& c = c64;
  auto row = [&](int s, int k, int r) {  // coefficient of shell r in moment s of family k
    const double x = (k == 0) ? S[s][r] : (k == 1) ? Q[s][r] : X[s][r];
    return (k == 3 && s >= 2) ? -x : x;
  };
  *t = AdjSplitTable<R>();
  for (int l = 0; l < 16; ++l) {
    const int s = l >> 2, k = l & 3;
    const bool half = l == 8 || l == 9 || l == 13;
    t->twice[l] = R(half ? 2 : 1);
    for (int r = 0; r < 4; ++r) {
      t->mom[r][l] = (R)(row(s, k, r) * (half ? 0.5 : 1.0));
      t->back[r][l] = (R)row(r, k, s);
      if (k == 0) t->inv_t[r][l] = (R)c.invS[r][s];
      if (k == 2) t->inv_t[r][l] = (R)c.invX[r][s];
      if (k == 3) t->inv_t[r][l] = (R)c.invY[r][s];
      if (k == 1 && (r & 1) == (s & 1)) t->inv_t[r][l] = (R)((s & 1) ? c.invP[r >> 1][s >> 1] : c.invQ[r >> 1][s >> 1]);
    }
    const int mo = moment[s][k];
    t->rate[l] = (mo >= 4) ? a.c.rate[mo] : R(0);
    t->wg[l] = (R)((k == 0) ? 1.0 : (k == 1) ? S[1][s] : X[0][s]);
    t->wl[l] = (k == 2) ? a.c.invX[s][1] : (k == 3) ? a.c.invY[s][1] : R(0);
    for (int q = 0; q < 4; ++q) t->lw[q][l] = a.c.lw[l][q];
    t->selfw[l] = a.selfw[l];
  }
  auto put = [&](int l, double r0, double r1, double x0, double x1, double y0, double y1, double e) {
    t->dr[0][l] = (R)r0; t->dr[1][l] = (R)r1;
    t->dx[0][l] = (R)x0; t->dx[1][l] = (R)x1;
    t->dy[0][l] = (R)y0; t->dy[1][l] = (R)y1;
    t->de[l] = (R)e;
  };
  put(1, -1, 0, 2, 0, -2, 0, 0);     // m4 = (jx^2 - jy^2) / rho
  put(5, -1, 0, 1, 0, 1, 0, 0);      // m5 = jx jy / rho
  put(6, 0.5, -1, 1, -1, -1, 0, 2);  // m6 = (e + p) ux
  put(7, 0.5, -1, -1, 0, 1, -1, 2);  // m7 = (e + p) uy
  put(10, -2, 6, 3, 0, -6, 0, 0);    // m8 = jx (ux^2 - 3 uy^2)
  put(11, -6, 2, 6, 0, 3, 0, 0);     // m9 = jy (3 ux^2 - uy^2)
  put(8, -2, 0, -1, 0, -1, 0, 4);    // m10 = 2 e^2 / rho - rho u^4 / 4 (its 3/4 u^4 apart)
  put(9, 2, -4, 4, -4, -4, -4, 6);   // m12 = w (ux^2 - uy^2)
  put(13, 2, -4, 2, -4, 2, -4, 6);   // m13 = w ux uy
  t->ga[6] = a.g[0]; t->gb[6] = a.g[1];    // A0 / s5 + A1 / s6
  t->ga[7] = a.g[1]; t->gb[7] = a.g[0];    // A2 / s6 + A3 / s5
  t->ga[1] = -a.g[2]; t->gb[1] = -a.g[4];  // -c6 A0 s7 / s5^2 - c7 A3 s8 / s5^2
  t->ga[5] = -a.g[3]; t->gb[5] = -a.g[5];  // -c6 A1 s7 / s6^2 - c7 A2 s8 / s6^2
}

}  // namespace
}  // namespace mrtlb
