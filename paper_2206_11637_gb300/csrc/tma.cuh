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

// Waits for the phase of this parity, a bounded number of tries (each of which
// suspends the thread for up to the hardware's time limit); false if they ran
// out.
constexpr int MBAR_TRIES = 1 << 20;
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
  unsigned done = 0;
  for (int k = 0; k < MBAR_TRIES && !done; ++k)
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
  return done != 0;
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
