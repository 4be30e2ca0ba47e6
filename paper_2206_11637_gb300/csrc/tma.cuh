// Tensor copies (TMA) into shared memory and the mbarriers they report to.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace pfl {

// Tensor maps of the current populations, (x, y, z, member), whose box is one
// tile of one plane with every member.
struct StepMaps {
  CUtensorMap h, g;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// One arrival (the thread that issues the copy) and the bytes it announces
// complete a phase.  Followed by a block barrier before anything uses them.
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ unsigned timer_ns() {  // wraps after 4.3 s
  unsigned t;
  asm volatile("mov.u32 %0, %globaltimer_lo;" : "=r"(t));
  return t;
}

// Waits for copy n (from 0; one in flight at a time) that reports to the barrier:
// it completes the n-th phase, of parity n & 1.  False once `limit` ns have passed
// without it; n < 0, no copy: true.  The limit is far above any copy's time, also
// on a GPU that is shared in time slices; the tries (each may suspend the thread for
// the hardware's own limit) end the wait should the timer stand still.  A block that
// gives up waits once more for the same copies, which may still be in flight,
// before its memory goes.
//
// The caller numbers the copies, and the wait past its first try is a function of its
// own, so that neither holds registers in the step: with counters and a 64-bit timer
// inline the D3Q27 bubble 128x384x128 took 519 us per step, now 501.
constexpr unsigned COPY_LIMIT_NS = 1000000000u;
constexpr int COPY_TRIES = 1 << 26;
static __device__ __noinline__ bool copy_wait_on(unsigned bar, unsigned parity, unsigned limit) {
  const unsigned t0 = timer_ns();
  for (int k = 0; k < COPY_TRIES && timer_ns() - t0 < limit; ++k)
    if (mbar_try(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ bool copy_wait(unsigned bar, int n, unsigned limit = COPY_LIMIT_NS) {
  if (n < 0 || mbar_try(bar, n & 1)) return true;
  return copy_wait_on(bar, n & 1, limit);
}

// The box at (x, y, z, w) of a rank-4 map into shared memory at dst.
__device__ __forceinline__ void tma4(unsigned dst, const CUtensorMap* m, int x, int y, int z, int w, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
          dst),
      "l"(m), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}

}  // namespace pfl
