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

// Waits for the phase of this parity; false once `limit` ns have passed without
// it.  The limit is far above any copy's time, also on a GPU that is shared in time
// slices; the tries (each may suspend the thread for the hardware's own limit) end
// the wait should the timer stand still.
constexpr unsigned long long MBAR_LIMIT_NS = 1000000000ull;
constexpr int MBAR_TRIES = 1 << 26;
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, unsigned long long limit = MBAR_LIMIT_NS) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = timer_ns();
  for (int k = 0; k < MBAR_TRIES && timer_ns() - t0 < limit; ++k)
    if (mbar_try(bar, parity)) return true;
  return false;
}

// An mbarrier and the copies that report to it, one in flight at a time: phase n
// is armed by the n-th copy and has parity n & 1.
struct CopyGate {
  unsigned bar;
  unsigned waited = 0;  // phases waited for
  __device__ __forceinline__ bool wait(unsigned long long limit = MBAR_LIMIT_NS) {
    return mbar_wait(bar, waited++ & 1, limit);
  }
  // After a wait that ran out, before the block's memory goes: the phase last
  // waited for once more, whose copy may still be in flight (true at once where it
  // has arrived, or where none was issued).
  __device__ __forceinline__ bool drain(unsigned long long limit = MBAR_LIMIT_NS) {
    return waited == 0 || mbar_wait(bar, (waited - 1) & 1, limit);
  }
};

// The box at (x, y, z, w) of a rank-4 map into shared memory at dst.
__device__ __forceinline__ void tma4(unsigned dst, const CUtensorMap* m, int x, int y, int z, int w, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
          dst),
      "l"(m), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}

}  // namespace pfl
