// Inline-PTX helpers for sm_103a: mbarriers, TMA tile loads, ex2.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace kqr {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase.  Gives up after max_polls polls (each
// try_wait itself suspends for a hardware-chosen interval), records
// kErrWaitTimeout in *err and returns false; the caller then stops its work and drains what is in flight.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, int* err,
                                                  uint32_t max_polls = (1u << 22)) {
  for (uint32_t i = 0; i < max_polls; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  atomicExch(err, 1);
  return false;
}

// 2-D tiled TMA load of box (x, y) of tensor map *tm into shared memory,
// completing transaction bytes on *bar.  x must be a multiple of 16 bytes /
// element size (every call here passes a multiple of 128 elements).
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// For CTAs that double-buffer column tiles, bars[0] for the row tile and bars[1 + (k & 1)] for column tile
// k: thread 0 calls it on its way out after a wait that gave up, so that the row tile's copy and the
// last two of the `issued` column tiles' have landed (bounded) before the CTA can end.  On the normal
// way out it has waited for each of them.
static __device__ __noinline__ void tile_drain(uint64_t* bars, int issued, int* err) {
  mbar_wait_bounded(&bars[0], 0, err);
  for (int k = issued > 2 ? issued - 2 : 0; k < issued; ++k)
    mbar_wait_bounded(&bars[1 + (k & 1)], (uint32_t)((k >> 1) & 1), err);
}

// The same for the MMAs of tiles k0 .. k1 - 1, committed to done[k & 1].
static __device__ __noinline__ void mma_drain(uint64_t* done, int k0, int k1, int* err) {
  for (int k = k0; k < k1; ++k) mbar_wait_bounded(&done[k & 1], (uint32_t)((k >> 1) & 1), err);
}

// Index of this thread's warp, the same register value in all its lanes: branches on it are uniform.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// True in one lane of a converged warp (the same one every time).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace kqr
