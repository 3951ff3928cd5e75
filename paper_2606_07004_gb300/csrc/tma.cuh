// TMA and mbarrier helpers (inline PTX) and tensor-map encoders shared by the
// sweep kernels (dia.cu, fix.cu).
#pragma once

#include "common.cuh"

namespace ld {

// Tensor maps over rows of 4-byte words: 2D (inner words x outer rows, rows
// `pitch` words apart), and the L x ny x nz grid of DiaInfo (box of box_inner
// words x bx x by x 1 points).  Points outside read as zero.
int tma_encode_ready();
int tma_encode_2d(CUtensorMap* map, const float* base, int inner, int outer, int pitch,
                  int box_inner, int box_outer);
int tma_encode_grid(CUtensorMap* map, const float* base, const DiaInfo& d, int inner, int pitch,
                    int box_inner, int bx, int by);

// A wait gives up after wait_ns of the global timer (2 s in normal use), or
// after kDiaWaitPolls polls whatever the timer says.
constexpr int kDiaWaitPolls = 1 << 24;
constexpr unsigned long long kDiaWaitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(phase)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for the barrier's phase to complete.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t phase,
                                                  unsigned long long wait_ns) {
  if (mbar_try_wait(bar, phase)) return true;
  const unsigned long long t0 = global_ns();
  for (int i = 0; i < kDiaWaitPolls; i += 32) {
    for (int k = 0; k < 32; ++k)
      if (mbar_try_wait(bar, phase)) return true;
    if (global_ns() - t0 > wait_ns) return false;
  }
  return false;
}
// 4D tiled copy of the box at (column, x, y, z) into shared memory.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c, int x,
                                            int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// 2D tiled copy of the box at (x = column, y = row) into shared memory.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

}  // namespace ld
