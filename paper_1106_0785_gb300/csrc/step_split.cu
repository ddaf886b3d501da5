// step_split.cu - the step of small grids: 16 lanes per node, one velocity each.
//
// A grid of a few thousand nodes has fewer nodes than the device has lanes,
// so its step takes as long as one thread's chain of instructions.  In FP64
// that chain is the whole cost: GB300 issues one FP64 instruction per 64
// cycles and SM sub-partition, however many lanes of the warp are active, and
// the one-thread-per-node kernel spends 508 of them a node.  Spread over the
// 16 lanes of half a warp, a node's step is 61.
//
// Lane l = 4 s + k holds velocity l of shell s.  Two butterfly stages inside
// the shell leave the lane with harmonic k of its shell (k = 0: S, 1: Q on the
// axis shells and P on the diagonal ones, 2: X, 3: Y); every moment is a
// combination of one harmonic family over the shells, so lane (s, k) forms
// moment s of family k from four lanes:
//            k = 0      1      2      3      (0-based moments)
//   s = 0      rho     m4     j_x    j_y
//       1       e      m5     m6     m7
//       2     m10/2   m12/2   m8     m9
//       3      m11    m13/2   m14    m15
// The equilibria are products of two lane-chosen operands, the halves above
// sparing their factors 2.  M^-1 goes back the same way.  The four
// neighbours' velocities take eleven additions in all: after the butterflies
// the sum over the shells is transposed, lane (s, k) ending with moment k of
// neighbour s (E, W, N, S), and one reciprocal serves all four.
//
// Walls and diffuse ghosts (REFILL) follow from the node's own moments and
// replace the neighbour's value before its velocity is formed.
#include "lanes.cuh"
#include "step_split.cuh"

namespace mrtlb {
namespace {

constexpr int kSplitThreads = 64;

// p = rho T and t = rho |u|^2
__device__ __forceinline__ double split_pressure(double, double jx, double jy, double e, double, double t) {
  return fma(-0.5, t, e);
}
__device__ __forceinline__ float split_pressure(float rho, float jx, float jy, float e, float ir, float) {
  return rho * temperature(rho, jx, jy, e, ir);  // (the compensated numerator)
}

template <typename R, bool REFILL>
__global__ void __launch_bounds__(kSplitThreads) step_split_kernel(const R* fin, R* __restrict__ fout, const Layout L,
                                                        const SplitTable<R>* __restrict__ tab, const R inv2dx,
                                                        const R inv2dy, const int version, const int modified,
                                                        R* keep, int* err) {
  const Lane<R> me(threadIdx.x);
  const int l = me.l, s = me.s, k = me.k;
  const int ni = L.i1 - L.i0;
  const int n = ni * (L.j1 - L.j0);
  const int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  const bool live = id < n;  // (the last half-warps repeat the last node: every lane takes part in the shuffles)
  const int t0 = live ? id : n - 1;
  const int i = L.i0 + t0 % ni, j = L.j0 + t0 / ni;
  // the constants load while the step before this one runs
  R cm[4], cf[4], ci[3], lw[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    cm[r] = tab->mom[r][l];
    lw[r] = tab->lw[r][l];
    if (REFILL) cf[r] = tab->full[r][l];
    if (r < 3) ci[r] = tab->inv[r][l];
  }
  const R rate = tab->rate[l], mod_a = tab->mod_a[l], mod_b = tab->mod_b[l];
  R wm[4];
  double wn[4], wd[4];
  if (REFILL) {
#pragma unroll
    for (int sd = 0; sd < 4; ++sd) {
      wm[sd] = tab->wall[sd][l];
      wn[sd] = tab->num[sd][l];
      wd[sd] = tab->inv_den[sd];
    }
  }
  after_previous();
  const R* at = fin + l * L.plane + L.node(i, j);
  const R f = at[0];
  R nb[4] = {at[1], at[-1], at[L.pitch], at[-L.pitch]};  // E, W, N, S

  const R m = me.moment(me.harmonic(f), cm);
  const R rho = from_lane(m, 0), e = from_lane(m, 4), jx = from_lane(m, 2), jy = from_lane(m, 3);
  R ir = R(0), vn = R(0);
  // after the butterflies: the sums over the shells of the neighbours' moments,
  // lane (s, k) ending with moment k (rho, -, j_x, j_y) of neighbour s
  auto neighbours = [&]() {
    R h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = me.harmonic(nb[q]);
    const bool odd = s & 1;
    const R a = (odd ? h[1] : h[0]) + across(odd ? h[0] : h[1], 4);
    const R b = (odd ? h[3] : h[2]) + across(odd ? h[2] : h[3], 4);
    const bool high = s >> 1;
    const R own = high ? b : a, oth = across(high ? a : b, 8);
    // (own: shells 2, 3 for high lanes, whose weight in j is 2)
    vn = (high ? own : oth) * (k == 0 ? R(1) : R(2)) + (high ? oth : own);
  };
  if (REFILL) {
    ir = split_recip(rho);
  } else {
    neighbours();
    const R rn = from_lane(vn, 4 * s);
    const R r = split_recip(k == 1 ? rho : rn);  // one reciprocal for the node and its neighbours
    ir = from_lane(r, 1);
    vn *= r;
  }
  const R ux = jx * ir, uy = jy * ir;
  const R t = jx * ux + jy * uy;
  const R p = split_pressure(rho, jx, jy, e, ir, t);

  R d = me.departure(m, rho, ir, jx, jy, e, ux, uy, t, p);
  if (version == 2 && l >= 14) {
    // m14 = rho ux (-4 + 10 T + 5 (ux^2 - uy^2)), m15 = rho uy (4 - 10 T + 5 (ux^2 - uy^2))
    const R T = p * ir, g = R(10) * T - R(4), w = R(5) * (ux * ux - uy * uy);
    d = m - (l == 14 ? jx * (w + g) : jy * (w - g));
  } else if (version == 3) {
    // rows 11, 14, 15 of M on rho / (2 pi T) exp(-|v - u|^2 / 2 T)
    const R T = p * ir, iT = split_recip(T);
    const R dx = R(vx_of(l)) - ux, dy = R(vy_of(l)) - uy;
    const R g = rho * (iT * R(0.15915494309189533576888376337251)) * expr(R(-0.5) * iT * (dx * dx + dy * dy));
    const R mg = me.moment(me.harmonic(g), cm);
    if (l == 12 || l >= 14) d = m - mg;
  }

  if (REFILL) {
    const R eq = (l == 0 || (l >= 2 && l <= 4)) ? m : m - d;  // (rho, j_x, j_y, e are their own equilibria)
#pragma unroll
    for (int sd = 0; sd < 4; ++sd) {
      R& b = nb[sd ^ 1];  // side order -x, +x, -y, +y; neighbours E, W, N, S
      const bool mine = beside_refilled(L, sd, i, j);
      if (L.bc[sd] == BC_WALL && __any_sync(kAll, mine)) {
        const R dm = (l == 0) ? R(0) : rho * wm[sd] - eq;  // (see wall_value)
        R h = R(0);
#pragma unroll
        for (int r = 0; r < 4; ++r) h += cf[r] * from_lane(dm, 4 * r + k);
        const R df = me.velocity(h);
        if (mine) b = f + df;
      } else if (L.bc[sd] == BC_DIFFUSE && __any_sync(kAll, mine)) {
        double num = wn[sd] * (double)f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) num += across(num, o);
        const double rw = num * wd[sd];
        const int vc = sd < 2 ? vx_of(l) : vy_of(l);
        const bool in = (sd & 1) ? vc < 0 : vc > 0;
        if (mine) b = in ? (R)(rw * tab->e64[sd][l]) : f;
      }
      // (for the adjoint, which reads the state with its walls)
      if (keep && live && mine)
        keep[l * L.plane + L.node(i, j) + (sd == 0 ? -1 : sd == 1 ? 1 : sd == 2 ? -(long long)L.pitch : L.pitch)] = b;
    }
    neighbours();
    vn *= split_recip(from_lane(vn, 4 * s));
  }

  R c = rate * d;
  if (modified) {
    // lanes (0, 2), (0, 3): d u / dx; (2, 2), (2, 3): d u / dy (before 1 / 2 d)
    const R g = vn - across(vn, 4);
    const bool sh = (l & 1) == 0;  // even lanes form the shear, odd ones the strain
    const R gx = from_lane(g, sh ? 2 : 3), gy = from_lane(g, sh ? 11 : 10);
    const R st = gx * inv2dx + (sh ? -(gy * inv2dy) : gy * inv2dy);
    // m6 += p (mod0 ux shear + mod1 uy strain), m7 += p (mod2 ux strain + mod3 uy shear)
    const R o = across(st, 1);
    c += p * (mod_a * (ux * st) + mod_b * (uy * o));
  }
  R h = ci[0] * from_lane(c, 4 * (k == 1 ? (s & 1) : 1) + k);
  h += ci[1] * from_lane(c, 4 * (k == 1 ? (s & 1) + 2 : 2) + k);
  h += ci[2] * from_lane(c, 12 + k);
  const R C = me.velocity(h);

  R inc = -C;
#pragma unroll
  for (int q = 0; q < 4; ++q) inc += lw[q] * (nb[q] - f);  // (as lw_update: a uniform region stays uniform)
  const R v = f + inc;
  if (!live) return;
  R* out = fout + L.node(i, j);
  out[l * L.plane] = v;
  const GhostTargets g = ghost_targets(L, i, j);
  if (g.any()) {
    const int mx = 4 * s + (me.axis ? (k & 1 ? k : k ^ 2) : k ^ 1);  // the mirrored velocities
    const int my = 4 * s + (me.axis ? (k & 1 ? k ^ 2 : k) : k ^ 3);
#pragma unroll
    for (int sd = 0; sd < 4; ++sd)
      if (g.w[sd]) out[(g.mir[sd] ? (sd < 2 ? mx : my) : l) * L.plane + g.off[sd]] = v;
  }
  if (l == 0 && (!(rho > R(0)) || !(p > R(0)))) atomicOr(err, ERRBIT_NONPHYSICAL);
}

}  // namespace

template <typename R>
void split_table(const Coef<R>& c, const Walls& w, SplitTable<R>* t) {
  static const double S[4][4] = {{1, 1, 1, 1}, {0.5, 1, 2, 4}, {0.125, 0.5, 2, 8}, {1, -4, 16, -64}};
  static const double X[4][4] = {{1, 1, 2, 2}, {0.5, 1, 4, 8}, {1, -2, 8, -16}, {1, -4, 32, -128}};
  static const double Q[4][4] = {{1, 0, 4, 0}, {0, 1, 0, 4}, {0.5, 0, 8, 0}, {0, 1, 0, 16}};
  static const int moment[4][4] = {{0, 4, 1, 2}, {3, 5, 6, 7}, {10, 12, 8, 9}, {11, 13, 14, 15}};  // [s][k]
  *t = SplitTable<R>();
  for (int l = 0; l < 16; ++l) {
    const int s = l >> 2, k = l & 3;
    for (int r = 0; r < 4; ++r) {
      const double x = (k == 0) ? S[s][r] : (k == 1) ? Q[s][r] : X[s][r];
      t->mom[r][l] = (R)((k == 3 && s >= 2) ? -x : x);
      // the lanes of moments 10, 12 and 13 hold halves of them
      if (k == 0) t->full[r][l] = c.invS[s][r] * R(r == 2 ? 2 : 1);
      if (k == 2) t->full[r][l] = c.invX[s][r];
      if (k == 3) t->full[r][l] = c.invY[s][r];
      if (k == 1 && (r & 1) == (s & 1))
        t->full[r][l] = ((s & 1) ? c.invP[s >> 1][r >> 1] : c.invQ[s >> 1][r >> 1]) * R(r >= 2 ? 2 : 1);
    }
    if (k == 1) {
      t->inv[0][l] = t->full[s & 1][l];
      t->inv[1][l] = t->full[(s & 1) + 2][l];
    } else {
      for (int r = 1; r < 4; ++r) t->inv[r - 1][l] = (k == 0 && r == 1) ? R(0) : t->full[r][l];
    }
    t->rate[l] = c.rate[moment[s][k]];
    for (int q = 0; q < 4; ++q) t->lw[q][l] = c.lw[l][q];
    for (int sd = 0; sd < 4; ++sd) {
      t->wall[sd][l] = (R)(w.m64[sd][moment[s][k]] * (l == 8 || l == 9 || l == 13 ? 0.5 : 1.0));
      t->e64[sd][l] = w.e64[sd][l];
      t->num[sd][l] = w.num[sd][l];
    }
  }
  for (int sd = 0; sd < 4; ++sd) t->inv_den[sd] = 1.0 / w.den[sd];
  t->mod_a[6] = c.mod[0];
  t->mod_b[6] = c.mod[1];
  t->mod_a[7] = c.mod[2];
  t->mod_b[7] = c.mod[3];
}

// The lines lie where another kernel takes over, us per step on GB300, 16 lanes per
// node / one thread.  FP64, which takes turns of two nodes a warp at 61 FP64
// instructions against rounds of 32 at 508 (version 1): 6000 nodes 15.6 / 18.7, 6400
// 18.9 / 18.5, version 2 17.2 / 19.1 and 20.8 / 18.9, version 3, whose exponentials
// it spreads over the lanes, 6800 28.2 / 29.6; with walls 7000 23.4 / 24.2, 7560 25.4 /
// 24.2, version 3 37.2 / 47.2; diffuse 6400 20.4 / 21.6, 7200 23.7 / 21.6.  FP32, bound
// by the length of one thread's chain, 1600 nodes 2.2 / 2.7 (tiles above the line 2.2),
// with walls 4000 3.45 / 3.5, diffuse 9000 4.96 / 6.5.  At the start of it all
// Sod 400 x 4 FP64 took 18.6 -> 5.7, Couette 4 x 200 FP64 28.6 -> 5.8 and FP32
// 4.8 -> 2.5, slip Couette 100 x 5 FP64 29.4 -> 5.9 and FP32 12.0 -> 3.1.
template <typename R>
bool use_split(const Layout& L, int version) {
  const bool wall = has_side(L, BC_WALL), diffuse = has_side(L, BC_DIFFUSE);
  const long long most = sizeof(R) == 4 ? (diffuse ? 10000 : wall ? 4000 : 2000)
                         : wall         ? (version == 3 ? 8000 : 7300)
                         : diffuse      ? 6500
                                        : (version == 3 ? 7000 : 6080);
  return (long long)(L.i1 - L.i0) * (L.j1 - L.j0) <= most;
}

template <typename R>
void launch_step_split(const R* fin, R* fout, const Layout& L, const Coef<R>& c, const SplitTable<R>* t, bool refill,
                       bool keep, int* err, cudaStream_t st) {
  const int ni = L.i1 - L.i0, nj = L.j1 - L.j0;
  if (ni <= 0 || nj <= 0) return;
  const unsigned grd = (unsigned)(((long long)ni * nj * 16 + kSplitThreads - 1) / kSplitThreads);
  const auto kernel = (refill && wall_count(L) > 0) ? step_split_kernel<R, true> : step_split_kernel<R, false>;
  // FP64 warps that share a sub-partition take turns, so blocks have to lie
  // evenly: set up early only up to two warps each (3200 nodes: 9.6 -> 14.5 us)
  const bool early = sizeof(R) == 4 || (long long)grd * (kSplitThreads / 32) <= 8LL * sm_count();
  launch_chained(early, kernel, grd, kSplitThreads, st, fin, fout, L, t, c.inv2dx, c.inv2dy, c.version, c.modified,
                 keep ? const_cast<R*>(fin) : nullptr, err);
}

#define MRTLB_INSTANTIATE(R)                                                                                   \
  template void split_table<R>(const Coef<R>&, const Walls&, SplitTable<R>*);                                  \
  template bool use_split<R>(const Layout&, int);                                                              \
  template void launch_step_split<R>(const R*, R*, const Layout&, const Coef<R>&, const SplitTable<R>*, bool, bool, int*, \
                                     cudaStream_t);
MRTLB_INSTANTIATE(float)
MRTLB_INSTANTIATE(double)

}  // namespace mrtlb
