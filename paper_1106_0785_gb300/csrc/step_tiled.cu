// step_tiled.cu - TMA-fed row-marching step kernel (the FP32 hot path):
// one CTA per (column strip, row segment) of a single grid.  The device
// side of the march lives in march.cuh.
#include <cuda.h>

#include <algorithm>
#include <cstddef>

#include "march_f64.cuh"
#include "march_pair.cuh"
#include "step_split.cuh"
#include "step_tiled.cuh"

namespace mrtlb {

namespace {

__global__ void __launch_bounds__(kRow64) step_f64_kernel(const __grid_constant__ CUtensorMap tmap,
                                                          double* __restrict__ fout, const Layout L,
                                                          const __grid_constant__ Coef<double> c, int* err,
                                                          const int seglen) {
  using SM = March64::SM;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int ja = L.j0 + blockIdx.y * seglen;
  const int jb = min(ja + seglen, L.j1);
  if (ja >= jb) return;  // uniform over the CTA
  March64 m;
  m.slots = reinterpret_cast<double*>(smem_raw);
  m.U = reinterpret_cast<double*>(smem_raw + SM::u_off);
  m.bars = reinterpret_cast<uint64_t*>(smem_raw + SM::bar_off);
  m.map = &tmap;
  m.fout = fout;
  m.err = err;
  m.L = L;
  m.t = threadIdx.x;
  m.kbase = 0;
  if (m.t == 0) {
    for (int s = 0; s < kSlot64; ++s) mbar_init(&m.bars[s], 1);
    mbar_fence_init();
  }
  __syncthreads();
  // strips start on multiples of BX so that every TMA box starts on a
  // 16-byte boundary (xoff - HL and BX are multiples of 16 bytes)
  if (m.segment(c, blockIdx.x * kRow64, ja, jb)) {
    if (m.t == 0) atomicOr(err, ERRBIT_TIMEOUT);
    m.drain();
  }
}

// FP32 with two nodes per thread (march_pair.cuh): BX columns, BX/2 threads,
// 254 registers, four CTAs per SM.  Measured alternatives on GB300: a launch
// bound of five CTAs (168 registers: three warps share an SM sub-partition's
// register file) was 7% slower, 64-column strips with eight one-warp CTAs
// 5% slower.
template <int BX, int NSLOT, int MINB>
__global__ void __launch_bounds__(BX / 2, MINB)
    step_pair_kernel(const __grid_constant__ CUtensorMap tmap, float* __restrict__ fout, const Layout L,
                     const __grid_constant__ Coef<P2> c, int* err, const int seglen, const bool once) {
  using SM = PairSmem<BX, NSLOT>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int ja = L.j0 + blockIdx.y * seglen;
  const int jb = min(ja + seglen, L.j1);
  if (ja >= jb) return;  // uniform over the CTA
  PairMarch<BX, NSLOT> m;
  m.once = once;
  m.slots = reinterpret_cast<float*>(smem_raw);
  m.U = reinterpret_cast<float*>(smem_raw + SM::u_off);
  m.bars = reinterpret_cast<uint64_t*>(smem_raw + SM::bar_off);
  m.map = &tmap;
  m.fout = fout;
  m.err = err;
  m.plane = L.plane;
  m.L = L;
  m.t = threadIdx.x;
  m.kbase = 0;
  if (m.t == 0) {
    for (int s = 0; s < NSLOT; ++s) mbar_init(&m.bars[s], 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (m.segment(c, blockIdx.x * BX, ja, jb)) {
    if (m.t == 0) atomicOr(err, ERRBIT_TIMEOUT);
    m.drain();
  }
}

// Self-test of the bounded wait: one thread waits on an mbarrier that no
// arrival completes; the wait gives up after its bound and the kernel flags
// ERRBIT_TIMEOUT, as a stalled march would.  No copy is in flight.
__global__ void wait_selftest_kernel(int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(&bar, 0)) atomicOr(err, ERRBIT_TIMEOUT);
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn get_encode() {
  static const EncodeFn fn = [] {  // thread-safe static initialisation
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return (EncodeFn)p;
    return (EncodeFn) nullptr;
  }();
  return fn;
}

// FP32 strips and ring
constexpr int kPairBX = 128, kPairSlots = 4, kPairBlocks = 4;

// The FP32 coefficient block with every constant in both lanes of a pair.
Coef<P2> pair_coef(const Coef<float>& c) {
  static_assert(offsetof(Coef<float>, version) % sizeof(float) == 0, "layout");
  constexpr int n = (int)(offsetof(Coef<float>, version) / sizeof(float));
  static_assert(offsetof(Coef<P2>, version) == n * sizeof(P2), "layout");
  Coef<P2> p;
  const float* src = &c.a1x;
  P2* dst = &p.a1x;
  for (int i = 0; i < n; ++i) dst[i] = P2(src[i]);
  p.version = c.version;
  p.modified = c.modified;
  return p;
}

}  // namespace

void plan_segments(const Layout& L, int target_ctas, TiledPlan* plan) {
  const int nj = L.j1 - L.j0;
  plan->nstrips = (L.i1 + plan->bx - 1) / plan->bx;
  if (plan->nstrips < 1) plan->nstrips = 1;
  int nseg = target_ctas / plan->nstrips;
  if (nseg < 1) nseg = 1;
  int seglen = (nj + nseg - 1) / nseg;
  if (seglen < 8) seglen = 8;
  if (seglen > nj) seglen = nj > 0 ? nj : 1;
  plan->seglen = seglen;
  plan->nseg = (nj + seglen - 1) / seglen;
}

// FP64: segments of the length with the least FP64 instructions on the busiest
// SM sub-partition (its warps take turns): a segment costs its rows and the two
// arrivals around them, and a pair of CTAs has a warp on each sub-partition.
// Returns whether that is less than the kernel it would replace takes, in FP64
// instructions of an SM's four sub-partitions with a warp each (38 ns), by
// equilibrium version: a row of the march; a round of 32 nodes on each
// sub-partition of the one-thread kernel, which with at most two warps an SM
// takes 0.92 of it; what refilled sides add to either, a wall launch before the
// march and a wall's arithmetic beside the plain kernel's nodes.  GB300, us per
// step, one thread per node / march: version 1 100 x 72 18.7 / 17.1, 160 x 120 20.9 /
// 30.8, 84 x 328 39.0 / 43.1, 256 x 256 76.2 / 55.2; version 3 49 x 176 29.5 / 32.3,
// 64 x 170 33.4 / 31.0, 515 x 103 96.3 / 111, 300 x 300 158 / 136; walls, version 1, 200 x
// 50 24.6 / 27.3, version 3 47.0 / 53.6.
static bool plan_f64(const Layout& L, int version, int nsm, TiledPlan* plan) {
  const int nj = std::max(1, L.j1 - L.j0);
  const long long n = (long long)(L.i1 - L.i0) * nj;
  const long long row = version == 3 ? 655 : version == 2 ? 338 : 323, round = version == 3 ? 840 : version == 2 ? 520 : 508;
  long long best = -1;
  for (int len = 1; len <= std::min(nj, 512); ++len) {
    const long long ctas = (long long)plan->nstrips * ((nj + len - 1) / len);
    const long long turns = ((ctas + nsm - 1) / nsm + 1) / 2;
    const long long cost = turns * (row * len + 110) + 40;
    // (segments of a few rows wait for their first copies in every turn)
    if (turns > 1 && len < std::min(4, nj)) continue;
    if (best < 0 || cost <= best) {
      best = cost;
      plan->seglen = len;
    }
  }
  plan->nseg = (nj + plan->seglen - 1) / plan->seglen;
  if (use_split<double>(L, version)) return false;  // (16 lanes per node: faster up to its line)
  const long long ctas = (long long)plan->nstrips * plan->nseg, turns = ((ctas + nsm - 1) / nsm + 1) / 2;
  long long march = turns * row * plan->seglen + (version == 3 ? 215 : 165) - (ctas <= nsm ? 40 : 0);
  const long long lanes = 128LL * nsm, rounds = (n + lanes - 1) / lanes;
  long long plain = 2 * n <= lanes ? round * 23 / 25 + 20 : round * rounds + 40;
  if (has_side(L, BC_WALL)) {
    march += version == 3 ? 550 : 230;
    // (with the walls' registers a last round that is nearly full, of three or more, takes one more)
    if (rounds > 2 && rounds * lanes - n < n / 32) plain += round;
    plain += version == 3 ? 450 + 25 * rounds : 145 + 15 * rounds;
  } else if (has_side(L, BC_DIFFUSE)) {
    march += 140;
    plain += 60 + 20 * rounds;
  }
  return march < plain;
}

int plan_tiled(const Layout& L, int version, int esize, void* f0, void* f1, TiledPlan* plan) {
  plan->ok = false;
  plan->esize = esize;
  EncodeFn enc = get_encode();
  if (!enc) return 1;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (nsm <= 0) nsm = 152;
  plan->bx = (esize == 4) ? kPairBX : kRow64;
  const int rc = encode_row_maps(L, esize, f0, f1, plan->bx, plan->map);
  if (rc) return rc;
  // the dynamic shared memory of the kernel launch_step_tiled will launch,
  // allowed in the current context (here: once per bind, on the bound
  // device, outside any stream capture), and its resident CTAs per SM
  const auto pair = step_pair_kernel<kPairBX, kPairSlots, kPairBlocks>;
  plan->smem = (esize == 4) ? PairSmem<kPairBX, kPairSlots>::bytes : March64::SM::bytes;
  const void* kernel = (esize == 4) ? (const void*)pair : (const void*)step_f64_kernel;
  int per_sm = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan->smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, esize == 4 ? kPairBX / 2 : kRow64, plan->smem) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return 4;
  }
  // One wave of resident CTAs; for the FP32 march the most waves, up to
  // four, whose segments keep at least kWaveRows rows (each wave then marches
  // a band of rows across the whole width).  Measured on GB300 (ms per step):
  // 4096 x 1024 0.0977 with one wave -> 0.0927 with two (segments of 54 ->
  // 27 rows); 2048 x 2048 0.0984 -> 0.0949 (two); 4096 x 1536 0.146 -> 0.136
  // (two) -> 0.1357 (three); 4096 x 2048 0.205 -> 0.184 (two) -> 0.179
  // (four); 4096 x 4096 0.382 (two) -> 0.356 (four); 3072 x 1024 0.0734 ->
  // 0.0720 (21 rows), but 3000 x 1000 0.0798 -> 0.0810 (20 rows, a ragged
  // last strip); a partial last wave (1.5 waves: 0.118 on 4096 x 1024)
  // leaves SMs idle.
  plan_segments(L, nsm * per_sm, plan);
  if (esize == 4) {
    constexpr int kWaveRows = 24;
    for (int waves = 4; waves >= 2; --waves) {
      TiledPlan more = *plan;
      plan_segments(L, waves * nsm * per_sm, &more);
      if (more.seglen >= kWaveRows) {
        plan->nstrips = more.nstrips;
        plan->nseg = more.nseg;
        plan->seglen = more.seglen;
        break;
      }
    }
  }
  // Where the two buffers together are larger than L2 and one of them fits, what a
  // step reads should make room for what it writes, which the next one reads.
  // GB300 (L2 129 MB), us per step without / with: 1501 x 701 (141 MB) 28.3 / 27.2,
  // 2048 x 600 (163 MB) 28.4 / 26.7, 2048 x 700 (190 MB) 33.0 / 31.4, 2048 x 800
  // (217 MB) 37.1 / 36.5; but 2048 x 900 (245 MB) 40.8 / 41.4, 4096 x 1024 87.1 / 98.8.
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
  const double both = 2.0 * 16.0 * (double)L.plane * esize;
  plan->once = esize == 4 && both > 1.0 * l2 && both <= 1.6 * l2;
  // FP32: a march of short segments (8 rows or more) is one wave whose time hardly
  // depends on the grid, the plain kernel's grows with the nodes; GB300, us per step,
  // plain / march: 1000 x 400 13.8 / 15.6, 1501 x 300 14.8 / 15.4, 1501 x 350 17.4 / 15.6;
  // version 3, whose plain kernel does less of it again, 1501 x 320 18.3 / 19.5, 1501 x
  // 350 20.1 / 19.2; walls, which the plain kernel works out beside its nodes or has
  // refilled first, 1000 x 400 17.0 / 17.3, 1501 x 280 17.9 / 17.3, version 3 1501 x 300
  // 21.5 / 22.0.
  if (esize == 4) {
    const long long nodes = (long long)(L.i1 - L.i0) * (L.j1 - L.j0);
    const bool refill = wall_count(L) > 0;
    plan->pays = plan->seglen >= kMinMarchRows ||
                 (refill ? nodes >= (version == 3 ? 3000LL : 2700LL) * nsm
                         : plan->nstrips * plan->nseg >= 3 * nsm && (version != 3 || nodes >= 3300LL * nsm));
  } else {
    plan->pays = plan_f64(L, version, nsm, plan);
  }
  plan->ok = true;
  return 0;
}

int encode_row_maps(const Layout& L, int esize, void* f0, void* f1, int bx, CUtensorMap out[2]) {
  EncodeFn enc = get_encode();
  if (!enc) return 1;
  const int hl = 16 / esize;
  if (((L.xoff - hl) * esize) % 16 != 0 || (bx * esize) % 16 != 0 || bx + 2 * hl > 256) return 3;
  const cuuint64_t dims[3] = {(cuuint64_t)L.pitch, (cuuint64_t)(L.ny + 2), 16};
  const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * esize, (cuuint64_t)L.plane * esize};
  const cuuint32_t box[3] = {(cuuint32_t)(bx + 2 * hl), 1, 16};
  const cuuint32_t estr[3] = {1, 1, 1};
  void* bufs[2] = {f0, f1};
  for (int b = 0; b < 2; ++b) {
    CUresult r = enc(&out[b], esize == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                     3, bufs[b], dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return 2;
  }
  return 0;
}

bool tiled_supported(const TiledPlan& plan) { return plan.ok; }

bool use_tiled(int which, const TiledPlan& plan) {
  if (!plan.ok) return false;
  if (which == MRTLB_KERNEL_PLAIN) return false;
  if (which == MRTLB_KERNEL_TILED) return true;
  return plan.pays;
}

template <typename R>
void launch_step_tiled(const TiledPlan& plan, int cur, const Layout& L, const Coef<R>& c, int* err,
                       cudaStream_t st, void* fout) {
  if (L.i1 <= L.i0 || L.j1 <= L.j0) return;
  const dim3 grd(plan.nstrips, plan.nseg);
  if constexpr (sizeof(R) == 4)
    step_pair_kernel<kPairBX, kPairSlots, kPairBlocks><<<grd, kPairBX / 2, plan.smem, st>>>(
        plan.map[cur], (float*)fout, L, pair_coef(c), err, plan.seglen, plan.once);
  else
    step_f64_kernel<<<grd, kRow64, plan.smem, st>>>(plan.map[cur], (double*)fout, L, c, err, plan.seglen);
}

void launch_wait_selftest(int* err, cudaStream_t st) { wait_selftest_kernel<<<1, 32, 0, st>>>(err); }

template void launch_step_tiled<float>(const TiledPlan&, int, const Layout&, const Coef<float>&, int*,
                                       cudaStream_t, void*);
template void launch_step_tiled<double>(const TiledPlan&, int, const Layout&, const Coef<double>&, int*,
                                        cudaStream_t, void*);

}  // namespace mrtlb
