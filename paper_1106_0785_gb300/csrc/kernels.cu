// kernels.cu - plain step kernel, boundary fills, layout conversion,
// equilibrium initialisation, macroscopic fields and conservation sums.
#include "kernels.cuh"

namespace mrtlb {

// ---------------------------------------------------------------------------
// Plain step: one thread per advanced node, neighbours read straight from
// global memory (L1/L2 serve the reuse).  The choice for grids too small for
// the row march, and the reference for it.
//
// REFILL: walls and diffuse ghosts are functions of the node beside them, so
// the node works them out from its own distributions and a step needs no
// launch before it that refills them in memory (whoever reads them there
// refills them first; and so do larger grids with walls, plain_walls_first).
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void velocity(const R g[16], R& ux, R& uy) {
  R rho, jx, jy, e;
  conserved(g, rho, jx, jy, e);
  const R r = recip(rho);
  ux = jx * r;
  uy = jy * r;
}
// Thread t takes advanced node t of the row-major enumeration of
// [i0, i1) x [j0, j1), so that every lane of a warp has a node whatever the
// grid's shape (a 4-column grid would leave 28 of 32 lanes idle under a
// 2D block, and FP64 arithmetic costs a warp the same with idle lanes).
template <typename R, bool REFILL>
__global__ void __launch_bounds__(128) step_plain_kernel(const R* __restrict__ fin, R* __restrict__ fout,
                                                         Layout L, Coef<R> c, Walls w, int* err) {
  const int ni = L.i1 - L.i0;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)ni * (L.j1 - L.j0)) return;
  const int i = L.i0 + (int)(t % ni);
  const int j = L.j0 + (int)(t / ni);
  const long long P = L.plane;
  const long long at = L.node(i, j);
  const long long E = at + 1, W = at - 1, N = at + L.pitch, S = at - L.pitch;
  after_previous();

  R f[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) f[q] = fin[q * P + at];
  R rho, jx, jy, e;
  conserved(f, rho, jx, jy, e);
  const R ir = recip(rho);
  const R ux = jx * ir, uy = jy * ir;
  const R T = temperature(rho, jx, jy, e, ir);

  R uxn[4], uyn[4], b[4][16];  // beyond sides -x, +x, -y, +y
  const long long nb[4] = {W, E, S, N};
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (REFILL && beside_refilled(L, s, i, j)) {
      refilled_value(c, w, L, s, f, b[s]);
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) b[s][q] = fin[q * P + nb[s]];
    }
    velocity(b[s], uxn[s], uyn[s]);
  }
  const R dux_dx = (uxn[1] - uxn[0]) * c.inv2dx, duy_dx = (uyn[1] - uyn[0]) * c.inv2dx;
  const R dux_dy = (uxn[3] - uxn[2]) * c.inv2dy, duy_dy = (uyn[3] - uyn[2]) * c.inv2dy;

  R C[16];
  collision(c, f, dux_dx, dux_dy, duy_dx, duy_dy, rho, ir, jx, jy, e, ux, uy, T, C);

  R vout[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    // (without REFILL read again, from L1, instead of held in registers)
    const R fE = REFILL ? b[1][q] : fin[q * P + E], fW = REFILL ? b[0][q] : fin[q * P + W];
    const R fN = REFILL ? b[3][q] : fin[q * P + N], fS = REFILL ? b[2][q] : fin[q * P + S];
    const R fn = lw_update(c, q, f[q], C[q], fE, fW, fN, fS);
    fout[q * P + at] = fn;
    vout[q] = fn;
  }
  const GhostTargets g = ghost_targets(L, i, j);
  if (g.any()) write_ghosts(g, P, vout, fout + at);
  if (!(rho > R(0)) || !(T > R(0))) atomicOr(err, ERRBIT_NONPHYSICAL);
}

// FP32 grids that the caches hold, without walls: a block of 128 threads takes a
// tile of nodes and shares their velocities, so that each is formed once (and
// those of the tile's rim by its first threads) instead of five times, and the
// neighbours' values, read for the update alone, are on their way meanwhile:
// 865 instructions a node instead of 950.  us per step on GB300, one thread per
// node / tile: 600 x 100 3.66 / 3.37, 300 x 300 5.16 / 4.87, 700 x 500 12.9 / 11.9,
// 1024 x 128 5.58 / 5.70.  (Two nodes per thread, as the march has them, would
// halve the instructions but are slower: one thread's chain is longer and half
// as many warps hide it, 600 x 100 3.92, 200 x 50 3.5 against 2.2.)
constexpr int kTileNodes = 128, kTileCells = (32 + 2) * (4 + 2);  // (the wider of the two tiles)
__global__ void __launch_bounds__(kTileNodes) step_tile_kernel(const float* __restrict__ fin, float* __restrict__ fout,
                                                               const Layout L, const __grid_constant__ Coef<float> c,
                                                               int* err) {
  __shared__ float su[2][kTileCells];
  const int TX = blockDim.x, TY = blockDim.y, tx = threadIdx.x, ty = threadIdx.y, SW = TX + 2;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int i = x0 + tx, j = y0 + ty;
  const long long P = L.plane;
  // the rim's cell this thread sees to: the rows below and above, then the columns beside
  const int h = ty * TX + tx;
  int hx = -2, hy = 0;
  if (h < TX) hx = h, hy = -1;
  else if (h < 2 * TX) hx = h - TX, hy = TY;
  else if (h < 2 * TX + TY) hx = -1, hy = h - 2 * TX;
  else if (h < 2 * TX + 2 * TY) hx = TX, hy = h - 2 * TX - TY;
  const bool rim = hx > -2 && x0 + hx <= L.nx && y0 + hy <= L.ny;
  const bool cell = i <= L.nx && j <= L.ny;  // (with the ghost beside the grid's last node)
  const bool node = i < L.nx && j < L.ny;
  after_previous();
  const float* at = fin + L.node(cell ? i : x0, cell ? j : y0);
  float f[16], g[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) f[q] = at[q * P];
  if (rim) {
    const float* r = fin + L.node(x0 + hx, y0 + hy);
#pragma unroll
    for (int q = 0; q < 16; ++q) g[q] = r[q * P];
  }
  float nE[16], nW[16], nN[16], nS[16];
  if (node) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      if (vx_of(q) != 0) nE[q] = at[q * P + 1], nW[q] = at[q * P - 1];
      if (vy_of(q) != 0) nN[q] = at[q * P + L.pitch], nS[q] = at[q * P - L.pitch];
    }
  }
  const NodeMac<float> m = node_macros(f);
  const int me = (ty + 1) * SW + tx + 1;
  su[0][me] = m.ux;
  su[1][me] = m.uy;
  if (rim) {
    float ux, uy;
    velocity(g, ux, uy);
    const int k = (hy + 1) * SW + hx + 1;
    su[0][k] = ux;
    su[1][k] = uy;
  }
  __syncthreads();
  if (!node) return;
  const float dux_dx = (su[0][me + 1] - su[0][me - 1]) * c.inv2dx, duy_dx = (su[1][me + 1] - su[1][me - 1]) * c.inv2dx;
  const float dux_dy = (su[0][me + SW] - su[0][me - SW]) * c.inv2dy, duy_dy = (su[1][me + SW] - su[1][me - SW]) * c.inv2dy;
  float C[16], v[16];
  collision(c, f, dux_dx, dux_dy, duy_dx, duy_dy, m.rho, m.ir, m.jx, m.jy, m.e, m.ux, m.uy, m.T, C);
  float* out = fout + L.node(i, j);
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    v[q] = lw_update(c, q, f[q], C[q], nE[q], nW[q], nN[q], nS[q]);
    out[q * P] = v[q];
  }
  const GhostTargets t = ghost_targets(L, i, j);
  if (t.any()) write_ghosts(t, P, v, out);
  if (!(m.rho > 0.0f) || !(m.T > 0.0f)) atomicOr(err, ERRBIT_NONPHYSICAL);
}
// The tile's width: 32 or 16, the wider first, where that leaves a quarter of
// the lanes idle at most; else 0.
static int tile_width(int ni) {
  for (int w = 32; w >= 16; w /= 2)
    if (4 * ni >= 3 * w * ((ni + w - 1) / w)) return w;
  return 0;
}

template <typename R>
void launch_step_plain(const R* fin, R* fout, const Layout& L, const Coef<R>& c, const Walls* w, int* err,
                       cudaStream_t st) {
  const int ni = L.i1 - L.i0, nj = L.j1 - L.j0;
  if (ni <= 0 || nj <= 0) return;
  // a grid small enough to leave SMs idle takes blocks of fewer threads
  // (the smallest power of two, at least 8, that covers it with one block
  // per SM), so that its latency-bound nodes spread over every SM
  const int nsm = sm_count();
  const long long n = (long long)ni * nj;
  int blk = 8;
  while (blk < 128 && (long long)blk * nsm < n) blk *= 2;
  const unsigned grd = (unsigned)((n + blk - 1) / blk);
  const bool refill = w && wall_count(L) > 0;
  if constexpr (sizeof(R) == 4) {
    const int tw = wall_count(L) > 0 ? 0 : tile_width(ni);
    if (tw) {
      const int th = kTileNodes / tw;
      launch_chained(true, step_tile_kernel, dim3((ni + tw - 1) / tw, (nj + th - 1) / th), dim3(tw, th), st, fin, fout, L,
                     c, err);
      return;
    }
  }
  const auto kernel = refill ? step_plain_kernel<R, true> : step_plain_kernel<R, false>;
  // (set up while the step before it runs: FP32 600 x 100 4.0 -> 3.7 us, 100 x 101
  // 2.74 -> 2.26; FP64 gains nothing)
  launch_chained(sizeof(R) == 4, kernel, grd, blk, st, fin, fout, L, c, refill ? *w : Walls{}, err);
}

// ---------------------------------------------------------------------------
// Boundaries.  Walls first (non-equilibrium extrapolation of Sec. IV A; the
// wall node takes f^eq(rho_a, u_w, T_w) + f_a - f^eq(rho_a, u_a, T_a) from
// its fluid neighbour a), then the ghost layer (periodic copy or
// zero-gradient outflow; behind a wall a copy keeps the ghost finite).
// ---------------------------------------------------------------------------
template <typename R>
__global__ void bc_walls_kernel(R* f, Layout L, Coef<R> c, Walls w) {
  wall_node(f, L, c, w, blockIdx.x * blockDim.x + threadIdx.x);
}

// One ghost value beside side s of a non-periodic side from the edge node
// `edge` (plane-0 address): outflow and walls copy it, reflect takes the
// mirrored plane, inflow the side's fixed equilibrium.
template <typename R>
__device__ __forceinline__ R side_ghost(const Walls& w, const Layout& L, int s, int q, const R* edge) {
  if (L.bc[s] == BC_INFLOW) return (R)(w.rho[s] * w.e64[s][q]);
  if (L.bc[s] == BC_REFLECT) return edge[(long long)(s < 2 ? mirror_x(q) : mirror_y(q)) * L.plane];
  return edge[(long long)q * L.plane];
}

// The ghost layer of f (plane q = blockIdx.y), diffuse sides excepted (the
// wall pass fills those).  only_inflow: just the inflow sides (buffers whose
// other ghosts the steps write).
template <typename R>
__global__ void bc_ghost_kernel(R* f, Layout L, Walls w, int only_inflow) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  const long long P = L.plane;
  R* fq = f + q * P;
  if (t < L.ny) {  // x sides, row j = t
    const int j = t;
    const long long row = (long long)(j + 1) * L.pitch;
    const long long first = row + L.xoff, last = row + L.xoff + L.nx - 1;
    if (L.bc[0] == BC_PERIODIC) {
      if (!only_inflow) {
        fq[first - 1] = fq[last];
        fq[last + 1] = fq[first];
      }
    } else {
      if ((!only_inflow && L.bc[0] != BC_DIFFUSE) || L.bc[0] == BC_INFLOW)
        fq[first - 1] = side_ghost(w, L, 0, q, f + first);
      if ((!only_inflow && L.bc[1] != BC_DIFFUSE) || L.bc[1] == BC_INFLOW)
        fq[last + 1] = side_ghost(w, L, 1, q, f + last);
    }
  }
  if (t < L.nx) {  // y sides, column i = t
    const int i = t;
    const long long first = (long long)1 * L.pitch + L.xoff + i;
    const long long last = (long long)L.ny * L.pitch + L.xoff + i;
    if (L.bc[2] == BC_PERIODIC) {
      if (!only_inflow) {
        fq[first - L.pitch] = fq[last];
        fq[last + L.pitch] = fq[first];
      }
    } else {
      if ((!only_inflow && L.bc[2] != BC_DIFFUSE) || L.bc[2] == BC_INFLOW)
        fq[first - L.pitch] = side_ghost(w, L, 2, q, f + first);
      if ((!only_inflow && L.bc[3] != BC_DIFFUSE) || L.bc[3] == BC_INFLOW)
        fq[last + L.pitch] = side_ghost(w, L, 3, q, f + last);
    }
  }
}

template <typename R>
void launch_walls(R* f, const Layout& L, const Coef<R>& c, const Walls& w, cudaStream_t st) {
  const int nwall = wall_count(L);
  if (nwall > 0) bc_walls_kernel<R><<<(nwall + 127) / 128, 128, 0, st>>>(f, L, c, w);
}

template <typename R>
void launch_bc(R* f, const Layout& L, const Coef<R>& c, const Walls& w, cudaStream_t st) {
  launch_walls<R>(f, L, c, w, st);
  const int n = (L.nx > L.ny) ? L.nx : L.ny;
  dim3 grd((n + 255) / 256, 16);
  bc_ghost_kernel<R><<<grd, 256, 0, st>>>(f, L, w, 0);
}

template <typename R>
void launch_inflow(R* f, const Layout& L, const Coef<R>& c, const Walls& w, cudaStream_t st) {
  bool any = false;
  for (int s = 0; s < 4; ++s) any |= (L.bc[s] == BC_INFLOW);
  if (!any) return;
  const int n = (L.nx > L.ny) ? L.nx : L.ny;
  dim3 grd((n + 255) / 256, 16);
  bc_ghost_kernel<R><<<grd, 256, 0, st>>>(f, L, w, 1);
}

// ---------------------------------------------------------------------------
// Dense [16][ny][nx] <-> padded layout.  A copy: 2 x the state's bytes.  The
// rows of all planes are numbered through (q ny + j); a block takes the same
// columns of kPackRows x blockDim.y of them, every load of a thread before its
// first store, V values to a load (16 bytes where the dense rows allow it,
// else one), and as many threads to a row as it fills.  4096 x 1024 in FP32 on
// GB300, mrtlb_set_f with its other launches: 221 -> 106 us (a value per thread
// and a block per piece of a row before); 1501 x 701, rows off the 16-byte
// grid: 80 -> 64 us.
// ---------------------------------------------------------------------------
constexpr int kPackThreads = 256, kPackRows = 4;
template <typename R, int V>
struct alignas(sizeof(R) * V) PackVec {
  R v[V];
};
template <typename R, int V>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const R* __restrict__ from, R* __restrict__ to, Layout L,
                                                            int to_padded) {
  using T = PackVec<R, V>;
  for (long long i = ((long long)blockIdx.y * blockDim.x + threadIdx.x) * V; i < L.nx;
       i += (long long)gridDim.y * blockDim.x * V) {
    long long src[kPackRows], dst[kPackRows];
    T x[kPackRows];
#pragma unroll
    for (int k = 0; k < kPackRows; ++k) {
      const int row = (blockIdx.x * kPackRows + k) * blockDim.y + threadIdx.y;  // q ny + j
      if (row >= 16 * L.ny) {
        src[k] = -1;
        continue;
      }
      const int q = row / L.ny, j = row - q * L.ny;
      const long long dense = (long long)row * L.nx + i, padded = q * L.plane + L.node(0, j) + i;
      src[k] = to_padded ? dense : padded;
      dst[k] = to_padded ? padded : dense;
      x[k] = *reinterpret_cast<const T*>(from + src[k]);
    }
#pragma unroll
    for (int k = 0; k < kPackRows; ++k)
      if (src[k] >= 0) *reinterpret_cast<T*>(to + dst[k]) = x[k];
  }
}

template <typename R>
static void launch_copy(const R* from, R* to, const R* dense, const Layout& L, int to_padded, cudaStream_t st) {
  constexpr int V = 16 / (int)sizeof(R);
  const bool wide = L.nx % V == 0 && ((uintptr_t)dense & 15) == 0;  // (padded rows start on 128 bytes)
  const int per_row = wide ? L.nx / V : L.nx;
  int bx = 1;
  while (bx < kPackThreads && bx < per_row) bx *= 2;
  const dim3 blk(bx, kPackThreads / bx);
  const int rows = kPackRows * (int)blk.y;
  const int pieces = (per_row - 1) / bx + 1;
  const dim3 grd((16 * L.ny + rows - 1) / rows, pieces < 65535 ? pieces : 65535);
  if (wide) pack_kernel<R, V><<<grd, blk, 0, st>>>(from, to, L, to_padded);
  else pack_kernel<R, 1><<<grd, blk, 0, st>>>(from, to, L, to_padded);
}

static int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 152LL * 32) b = 152LL * 32;
  if (b < 1) b = 1;
  return (int)b;
}

template <typename R>
void launch_pack(const R* dense, R* padded, const Layout& L, cudaStream_t st) {
  launch_copy<R>(dense, padded, dense, L, 1, st);
}
template <typename R>
void launch_unpack(const R* padded, R* dense, const Layout& L, cudaStream_t st) {
  launch_copy<R>(padded, dense, dense, L, 0, st);
}

// ---------------------------------------------------------------------------
// f = M^-1 f^eq(rho, u, T), computed in FP64.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void init_eq_kernel(const double* __restrict__ rho_in, const double* __restrict__ ux_in,
                               const double* __restrict__ uy_in, const double* __restrict__ T_in,
                               R* __restrict__ f, Layout L, Coef<double> c) {
  const long long n = (long long)L.ny * L.nx;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    const double rho = rho_in[t], ux = ux_in[t], uy = uy_in[t], T = T_in[t];
    const double e = rho * (T + 0.5 * (ux * ux + uy * uy));
    double eq[16], g[16];
    equilibrium(c, rho, 1.0 / rho, rho * ux, rho * uy, e, ux, uy, T, eq);
    inverse_full(c, eq, g);
    const long long at = L.node(i, j);
#pragma unroll
    for (int q = 0; q < 16; ++q) f[q * L.plane + at] = (R)g[q];
  }
}

template <typename R>
void launch_init_eq(const double* rho, const double* ux, const double* uy, const double* T, R* f,
                    const Layout& L, const Coef<double>& c64, cudaStream_t st) {
  if constexpr (sizeof(R) == 4) {
    if (launch_init_eq_df(rho, ux, uy, T, f, L, c64, st)) return;
  }
  const long long n = (long long)L.ny * L.nx;
  init_eq_kernel<R><<<grid_for(n, 128), 128, 0, st>>>(rho, ux, uy, T, f, L, c64);
}

// ---------------------------------------------------------------------------
// rho, u, T in FP64 (Sec. II, R = 1).
// ---------------------------------------------------------------------------
// Moment sums in the storage precision (FP32 states: the same recovery as
// the step, FP32 sums and the compensated temperature numerator), outputs
// in FP64.
template <typename R>
__global__ void macros_kernel(const R* __restrict__ f, double* rho_o, double* ux_o, double* uy_o,
                              double* T_o, Layout L) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= L.nx) return;
  const long long t = (long long)j * L.nx + i;
  const long long at = L.node(i, j);
  R g[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) g[q] = f[q * L.plane + at];
  R rho, jx, jy, e;
  conserved(g, rho, jx, jy, e);
  const R ir = recip(rho);
  if (rho_o) rho_o[t] = (double)rho;
  if (ux_o) ux_o[t] = (double)(jx * ir);
  if (uy_o) uy_o[t] = (double)(jy * ir);
  if (T_o) T_o[t] = (double)temperature(rho, jx, jy, e, ir);
}

template <typename R>
void launch_macros(const R* f, double* rho, double* ux, double* uy, double* T, const Layout& L,
                   cudaStream_t st) {
  dim3 grd((L.nx + 127) / 128, L.ny);
  macros_kernel<R><<<grd, 128, 0, st>>>(f, rho, ux, uy, T, L);
}

// ---------------------------------------------------------------------------
// Conservation sums and the max |T - T_prev| residual of an FP64 state (of an
// FP32 one: start.cu).  Warp shuffles, then one atomic per warp.
// ---------------------------------------------------------------------------
__global__ void reduce_kernel(const double* __restrict__ f, double* acc, double* Tprev, int have_prev,
                              Layout L) {
  const long long n = (long long)L.ny * L.nx;
  double s0 = 0, s1 = 0, s2 = 0, s3 = 0, mx = 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    const long long at = L.node(i, j);
    double g[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) g[q] = f[q * L.plane + at];
    double rho, jx, jy, e;
    conserved(g, rho, jx, jy, e);
    s0 += rho; s1 += jx; s2 += jy; s3 += e;
    const double T = temperature(rho, jx, jy, e, 1.0 / rho);
    if (have_prev) {
      const double d = fabs(T - Tprev[t]);
      mx = (d > mx || d != d) ? d : mx;
    }
    Tprev[t] = T;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    s3 += __shfl_xor_sync(0xffffffffu, s3, o);
    const double m = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = (m > mx || m != m) ? m : mx;
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(acc + 0, s0);
    atomicAdd(acc + 1, s1);
    atomicAdd(acc + 2, s2);
    atomicAdd(acc + 3, s3);
    // non-negative doubles order like their bit patterns; NaN maps above inf
    atomicMax((unsigned long long*)(acc + 4), (unsigned long long)__double_as_longlong(mx));
  }
}

template <typename R>
void launch_reduce(const R* f, double* acc, double* Tprev, int have_prev, const Layout& L,
                   cudaStream_t st) {
  if constexpr (sizeof(R) == 4) {
    launch_reduce_f32(f, acc, Tprev, have_prev, L, st);
  } else {
    const long long n = (long long)L.ny * L.nx;
    reduce_kernel<<<grid_for(n, 256), 256, 0, st>>>(f, acc, Tprev, have_prev, L);
  }
}

#define MRTLB_INSTANTIATE(R)                                                                     \
  template void launch_step_plain<R>(const R*, R*, const Layout&, const Coef<R>&, const Walls*,   \
                                     int*, cudaStream_t);                                        \
  template void launch_bc<R>(R*, const Layout&, const Coef<R>&, const Walls&, cudaStream_t); \
  template void launch_walls<R>(R*, const Layout&, const Coef<R>&, const Walls&, cudaStream_t); \
  template void launch_inflow<R>(R*, const Layout&, const Coef<R>&, const Walls&, cudaStream_t); \
  template void launch_pack<R>(const R*, R*, const Layout&, cudaStream_t);                       \
  template void launch_unpack<R>(const R*, R*, const Layout&, cudaStream_t);                     \
  template void launch_init_eq<R>(const double*, const double*, const double*, const double*,    \
                                  R*, const Layout&, const Coef<double>&, cudaStream_t);         \
  template void launch_macros<R>(const R*, double*, double*, double*, double*, const Layout&,    \
                                 cudaStream_t);                                                  \
  template void launch_reduce<R>(const R*, double*, double*, int, const Layout&, cudaStream_t);

MRTLB_INSTANTIATE(float)
MRTLB_INSTANTIATE(double)

}  // namespace mrtlb
