// march_f64.cuh - the FP64 row march.
//
// Same pipeline as march_pair.cuh (a CTA per strip of BX columns and segment of
// rows; rows by TMA boxes into an NSLOT ring with bounded waits), one node per
// thread.  What bounds it is the FP64 pipe: GB300 issues an FP64 instruction
// per 64 cycles and SM sub-partition, so loads, shared memory and registers
// are free beside it and only the FP64 instructions count, 307 a node:
//   * a row's harmonics, moments and macroscopic state are formed once, when it
//     arrives, and carried in registers to its update an iteration later;
//   * u of the strip's two halo columns takes the lanes of one warp, sixteen a
//     column (a thread each would cost that warp a whole node's instructions
//     for two lanes' sake);
//   * m - m^eq is formed as fused multiply-adds from the moment on, the rates
//     are folded into M^-1 (CoefFold), 1/rho is Newton's iteration.
// (The Lax-Wendroff increment from the values' own weights instead of their
// differences would save 32 of them, but moves a uniform region by a last place
// at larger Courant numbers: see lw_update.)
// Before, 472 a node. GB300, ms per step: 4096 x 1024 3.18 -> 2.46, 1024 x 256
// 0.225 -> 0.177, 600 x 100 0.076 (one thread per node) -> 0.055; 16 grids of the
// batch 2.71 -> 2.14.
#pragma once

#include "lanes.cuh"
#include "march.cuh"

namespace mrtlb {
namespace {

constexpr int kRow64 = 64;   // columns of a strip
constexpr int kSlot64 = 4;   // rows in flight

// Macroscopic state and harmonics of a node.
struct Node64 {
  double rho, ir, jx, jy, e, ux, uy, p, t;  // p = rho T, t = rho |u|^2
  Harm<double> h;
};
__device__ __forceinline__ void harmonics64(const double f[16], Harm<double>& h) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const double p02 = f[4 * s] + f[4 * s + 2], p13 = f[4 * s + 1] + f[4 * s + 3];
    const double m02 = f[4 * s] - f[4 * s + 2], m13 = f[4 * s + 1] - f[4 * s + 3];
    h.S[s] = p02 + p13;
    if (s & 1) {
      h.X[s] = m02 - m13;
      h.Y[s] = m02 + m13;
      h.P[s >> 1] = p02 - p13;
    } else {
      h.X[s] = m02;
      h.Y[s] = m13;
      h.Q[s >> 1] = p02 - p13;
    }
  }
}
__device__ __forceinline__ void node64(const double f[16], Node64& n) {
  harmonics64(f, n.h);
  conserved_h(n.h, n.rho, n.jx, n.jy, n.e);
  n.ir = split_recip(n.rho);
  n.ux = n.jx * n.ir;
  n.uy = n.jy * n.ir;
  n.t = fma(n.jy, n.uy, n.jx * n.ux);
  n.p = fma(-0.5, n.t, n.e);
}

// dt C of a node from its state and the shear and strain of u.
__device__ __forceinline__ void collision64(const Coef<double>& c, const Node64& n, double shear, double strain,
                                            double C[16]) {
  const Harm<double>& h = n.h;
  const double ux = n.ux, uy = n.uy, x2 = ux * ux, y2 = uy * uy, xy = ux * uy, u2 = x2 + y2, d2 = x2 - y2;
  const double w2 = fma(3.0, n.e, -n.t), ep = n.e + n.p;  // 3 e - rho u^2, e + p
  // m - m^eq (d13: half of it)
  const double d4 = fma(n.jy, uy, fma(-n.jx, ux, fma(4.0, h.Q[1], h.Q[0])));
  const double d5 = fma(-n.jx, uy, fma(4.0, h.P[1], h.P[0]));
  double d6 = fma(0.5, h.X[0], h.X[1]), d7 = fma(0.5, h.Y[0], h.Y[1]);
  d6 = fma(-ep, ux, fma(8.0, h.X[3], fma(4.0, h.X[2], d6)));
  d7 = fma(-ep, uy, fma(8.0, h.Y[3], fma(4.0, h.Y[2], d7)));
  double d8 = fma(-16.0, h.X[3], fma(8.0, h.X[2], fma(-2.0, h.X[1], h.X[0])));
  double d9 = fma(16.0, h.Y[3], fma(-8.0, h.Y[2], fma(2.0, h.Y[1], -h.Y[0])));
  d8 = fma(-n.jx, fma(-3.0, y2, x2), d8);
  d9 = fma(-n.jy, fma(3.0, x2, -y2), d9);
  double d10 = fma(16.0, h.S[3], fma(4.0, h.S[2], fma(0.25, h.S[0], h.S[1])));
  d10 = fma(0.25 * n.t, u2, fma(-(n.e + n.e), n.e * n.ir, d10));
  double d11 = fma(-64.0, h.S[3], fma(16.0, h.S[2], fma(-4.0, h.S[1], h.S[0])));
  const double d12 = fma(-(w2 + w2), d2, fma(16.0, h.Q[1], h.Q[0]));
  const double d13 = fma(-w2, xy, fma(16.0, h.P[1], h.P[0]));
  double d14 = fma(-128.0, h.X[3], fma(32.0, h.X[2], fma(-4.0, h.X[1], h.X[0])));
  double d15 = fma(128.0, h.Y[3], fma(-32.0, h.Y[2], fma(4.0, h.Y[1], -h.Y[0])));
  if (c.version != 1) {
    double eq[16];
    equilibrium(c, n.rho, n.ir, n.jx, n.jy, n.e, ux, uy, n.p * n.ir, eq);
    d11 -= eq[11];
    d14 -= eq[14];
    d15 -= eq[15];
  }
  double c6 = c.rate[6] * d6, c7 = c.rate[7] * d7;
  if (c.modified) {
    const double px = n.p * ux, py = n.p * uy;
    c6 = fma(c.mod[0], px * shear, fma(c.mod[1], py * strain, c6));
    c7 = fma(c.mod[2], px * strain, fma(c.mod[3], py * shear, c7));
  }
  double S[4], X[4], Y[4], Q[2], P[2];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    S[s] = fma(c.fS[s][1], d11, c.fS[s][0] * d10);
    X[s] = fma(c.fX[s][1], d14, fma(c.fX[s][0], d8, c.invX[s][1] * c6));
    Y[s] = fma(c.fY[s][1], d15, fma(c.fY[s][0], d9, c.invY[s][1] * c7));
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    Q[s] = fma(c.fQ[s][1], d12, c.fQ[s][0] * d4);
    P[s] = fma(c.fP[s][1], d13, c.fP[s][0] * d5);
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const double qp = (s & 1) ? P[s >> 1] : Q[s >> 1];
    const double sp = S[s] + qp, sm = S[s] - qp;
    const double a = (s & 1) ? X[s] + Y[s] : X[s], b = (s & 1) ? Y[s] - X[s] : Y[s];
    C[4 * s + 0] = sp + a;
    C[4 * s + 2] = sp - a;
    C[4 * s + 1] = sm + b;
    C[4 * s + 3] = sm - b;
  }
}

struct March64 {
  static constexpr int BX = kRow64, NSLOT = kSlot64;
  using SM = Smem<double, BX, NSLOT>;
  double* slots;
  double* U;
  uint64_t* bars;
  const CUtensorMap* map;
  double* fout;
  int* err;
  int t, x, boxx, r_first, r_last, issued_to, kbase;
  bool active;
  Layout L;

  __device__ __forceinline__ int k(int r) const { return kbase + r - r_first; }
  __device__ __forceinline__ const double* slot(int r) const { return slots + (k(r) & (NSLOT - 1)) * SM::SLOT; }
  __device__ __forceinline__ double* urow(int r) const { return U + (k(r) & 3) * SM::UROW; }
  __device__ __forceinline__ bool ready(int r) const {
    return mbar_wait(&bars[k(r) & (NSLOT - 1)], (uint32_t)((k(r) / NSLOT) & 1));
  }
  __device__ __forceinline__ void issue(int r) {
    const int s = k(r) & (NSLOT - 1);
    mbar_expect_tx(&bars[s], (uint32_t)SM::slot_bytes);
    tma_load_row(slots + s * SM::SLOT, map, boxx, r + 1, &bars[s]);
  }
  // Row r of the thread's column into f, its state into n, its u (and that of
  // the strip's two halo columns) to the ring.
  __device__ __forceinline__ void arrive(int r, double f[16], Node64& n) const {
    const double* sl = slot(r);
    double* u = urow(r);
#pragma unroll
    for (int q = 0; q < 16; ++q) f[q] = sl[q * SM::BW + SM::HL + t];
    node64(f, n);
    u[t + 1] = n.ux;
    u[(BX + 2) + t + 1] = n.uy;
    if (t < 32) {  // lanes 0-15: column x0 - 1, lanes 16-31: x0 + BX; a velocity each
      const int l = t & 15, right = t >> 4;
      const double v = sl[l * SM::BW + (right ? SM::HL + BX : SM::HL - 1)];
      const bool axis = (l & 4) == 0;
      const int kk = l & 3;
      // shell sums and differences by two butterflies: k = 0 S, 2 X, 3 Y
      double o = __shfl_xor_sync(0xffffffffu, v, 2), h = (kk < 2) ? v + o : o - v;
      o = __shfl_xor_sync(0xffffffffu, h, 1);
      if (!axis && kk == 2) o = -o;
      h += (axis && kk >= 2) ? 0.0 : o;
      h += __shfl_xor_sync(0xffffffffu, h, 4);
      o = __shfl_xor_sync(0xffffffffu, h, 8);
      // shells 2 and 3 count twice in j
      const bool high = l & 8;
      h = fma((kk == 0) ? 1.0 : 2.0, high ? h : o, high ? o : h);
      const double rho = __shfl_sync(0xffffffffu, h, 0, 16), w = h * split_recip(rho);
      if (l == 2) u[right ? BX + 1 : 0] = w;
      if (l == 3) u[(BX + 2) + (right ? BX + 1 : 0)] = w;
    }
  }
  // Output row j: fp holds row j - 1, nc the state of row j; nn receives that
  // of row j + 1.  Returns true if the CTA must stop (a wait expired).
  __device__ __forceinline__ bool row(int j, const Coef<double>& c, double fp[16], const Node64& nc, Node64& nn) {
    const bool bad = !ready(j + 1);
    if (__syncthreads_or(bad)) return true;
    if (t == 0 && issued_to < r_last) {  // the slot of row j - 1 is free
      fence_proxy_async();
      ++issued_to;
      issue(issued_to);
    }
    double fn[16];
    arrive(j + 1, fn, nn);
    const double* sc = slot(j);
    const double* u = urow(j);
    const double* up = urow(j - 1);
    const double* uy = u + (BX + 2);
    const double shear = (u[t + 2] - u[t]) * c.inv2dx - (nn.uy - up[(BX + 2) + t + 1]) * c.inv2dy;
    const double strain = (uy[t + 2] - uy[t]) * c.inv2dx + (nn.ux - up[t + 1]) * c.inv2dy;
    double C[16];
    collision64(c, nc, shear, strain, C);
    double* out = fout + L.node(x, j);
    double v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const double* s = sc + q * SM::BW + SM::HL + t;
      const double f = s[0];
      double d = -C[q];
      if (vx_of(q) != 0) d = fma(c.lw[q][1], s[-1] - f, fma(c.lw[q][0], s[1] - f, d));
      if (vy_of(q) != 0) d = fma(c.lw[q][3], fp[q] - f, fma(c.lw[q][2], fn[q] - f, d));
      v[q] = f + d;
      if (active) out[q * L.plane] = v[q];
      fp[q] = f;
    }
    if (active) {
      const GhostTargets g = ghost_targets(L, x, j);
      if (g.any()) write_ghosts(g, L.plane, v, out);
      if (!(nc.rho > 0.0) || !(nc.p > 0.0)) atomicOr(err, ERRBIT_NONPHYSICAL);
    }
    return false;
  }
  // Advance rows [ja, jb) of the strip starting at column x0 (a multiple of
  // BX); rows ja-1 .. jb stream in.  Returns true if a wait expired (the CTA
  // agreed to stop).  Leaves kbase past the rows it streamed.
  __device__ __forceinline__ bool segment(const Coef<double>& c, int x0, int ja, int jb) {
    x = x0 + t;
    active = x >= L.i0 && x < L.i1;
    boxx = L.xoff + x0 - SM::HL;
    r_first = ja - 1;
    r_last = jb;
    if (t == 0)
      for (int kk = 0; kk < NSLOT && r_first + kk <= r_last; ++kk) issue(r_first + kk);
    issued_to = min(r_first + NSLOT - 1, r_last);
    double fp[16], f[16];
    Node64 nc, nn;
    bool bad = !ready(r_first);
    arrive(r_first, fp, nn);
    bad |= !ready(ja);
    arrive(ja, f, nc);
    bool stopped = __syncthreads_or(bad);
    for (int j = ja; !stopped && j < jb; ++j) {
      if ((stopped = row(j, c, fp, nc, nn))) break;
      nc = nn;
    }
    if (!stopped) kbase += r_last - r_first + 1;
    return stopped;
  }
  // after a stop: let copies still in flight land before the CTA's smem goes
  // away (the latest copy of each slot is the only one that can be pending)
  __device__ __forceinline__ void drain() {
    if (t == 0)
      for (int r = max(r_first, issued_to - NSLOT + 1); r <= issued_to; ++r) (void)ready(r);
    __syncthreads();
  }
};

}  // namespace
}  // namespace mrtlb
