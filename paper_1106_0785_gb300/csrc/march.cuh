// march.cuh - what the row marches share (march_pair.cuh in FP32, march_f64.cuh
// in FP64, adjoint_march.cuh): bounded mbarrier waits, the row loads and the
// shared-memory layout.
//
// A CTA owns a strip of BX columns and advances a segment of rows of one grid.
// For output row j it needs f at (x, j-1), (x, j), (x, j+1) and (x+-1, j), and
// u at the four cross neighbours, which is formed once per node when its row
// arrives and kept in a 4-row shared ring.  Rows arrive through
// cp.async.bulk.tensor (one 3D box = all 16 planes of one row plus a 16-byte
// halo on each side) into NSLOT slots, each with an mbarrier; thread 0 refills
// the slot of row j-1 once every thread is past the barrier of iteration j.
// Slot phases run on across the segments a persistent CTA takes in turn
// (kbase counts the rows it has streamed so far).
//
// Every mbarrier wait is bounded (about 2 s of wall clock, read from the
// global timer): on expiry the CTA agrees (barrier-or) to stop and the
// caller flags ERRBIT_TIMEOUT and drains the copies still in flight.
#pragma once

#include <cuda.h>

#include "kernels.cuh"

namespace mrtlb {
namespace {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s
constexpr unsigned kSuspendHintNs = 1000000u;                // 1 ms per poll

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// one poll; the thread may sleep up to the hint waiting for the phase
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendHintNs)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait; true when the phase completed
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_test(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (true) {
    if (mbar_test(bar, parity)) return true;
    if (global_ns() - t0 > kWaitLimitNs) return false;
  }
}
__device__ __forceinline__ void tma_load_row(void* dst, const CUtensorMap* map, int x, int y,
                                             uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(0), "r"(smem_u32(bar))
      : "memory");
}
// the same, the lines to leave L2 before others (a row that is read once)
__device__ __forceinline__ void tma_load_row_once(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(0), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

template <typename R, int BX, int NSLOT>
struct Smem {
  static_assert((NSLOT & (NSLOT - 1)) == 0 && NSLOT >= 4, "NSLOT: power of two >= 4");
  static constexpr int HL = 16 / (int)sizeof(R);  // halo columns either side
  static constexpr int BW = BX + 2 * HL;          // box width (elements)
  static constexpr int SLOT = 16 * BW;            // elements per slot
  static constexpr int UROW = 2 * (BX + 2);       // u_x, u_y of one row incl. halo
  static constexpr size_t slot_bytes = (size_t)SLOT * sizeof(R);
  static constexpr size_t u_off = (size_t)NSLOT * slot_bytes;
  static constexpr size_t u_bytes = (size_t)4 * UROW * sizeof(R);
  static constexpr size_t bar_off = (u_off + u_bytes + 15) & ~(size_t)15;
  static constexpr size_t bytes = bar_off + NSLOT * sizeof(uint64_t);
};

}  // namespace
}  // namespace mrtlb
