"""The waits of the tensor-copy step: a copy that does not arrive ends a wait at its limit, and the
block waits once more for the same copy before it leaves.

The waits (csrc/tma.cuh) run in a kernel of their own, whose copy is withheld, or issued only
after the first wait has run out; no copy is in flight when a block that gave up ends.
"""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

KERNEL = r"""
#include "tma.cuh"
using namespace pfl;
// res: first wait, its ns, drain, its ns, drain of a barrier without copies, its ns
__global__ void k_waits(const int* src, int late, unsigned long long limit, unsigned long long* res) {
  __shared__ unsigned long long mbar[2];
  __shared__ __align__(16) int dst[4];
  CopyGate a{smem_u32(mbar)}, b{smem_u32(mbar + 1)};
  if (threadIdx.x == 0) {
    mbar_init(a.bar);
    mbar_init(b.bar);
    mbar_expect(a.bar, 16);
  }
  __syncthreads();
  const unsigned long long t0 = timer_ns();
  const bool w = a.wait(limit);
  const unsigned long long t1 = timer_ns();
  __syncthreads();
  if (late && threadIdx.x == 0)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], 16, [%2];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(a.bar) : "memory");
  const unsigned long long t2 = timer_ns();
  const bool d = a.drain(limit);
  const unsigned long long t3 = timer_ns();
  const bool e = b.drain(limit);
  const unsigned long long t4 = timer_ns();
  if (threadIdx.x == 0) {
    const unsigned long long v[7] = {w, t1 - t0, d, t3 - t2, e, t4 - t3, d ? (unsigned long long)dst[0] : 0};
    for (int k = 0; k < 7; ++k) res[k] = v[k];
  }
}
extern "C" int run_waits(int late, unsigned long long limit, unsigned long long* out) {
  int *src, one[4] = {41, 0, 0, 0};
  unsigned long long* res;
  if (cudaMalloc(&src, 16) != cudaSuccess || cudaMalloc(&res, 56) != cudaSuccess) return 1;
  cudaMemcpy(src, one, 16, cudaMemcpyHostToDevice);
  k_waits<<<1, 64>>>(src, late, limit, res);
  const cudaError_t e = cudaMemcpy(out, res, 56, cudaMemcpyDeviceToHost);
  cudaFree(src);
  cudaFree(res);
  return (int)e;
}
"""
MS = 1000000


@pytest.fixture(scope="module")
def waits(tmp_path_factory):
    from paper_2206_11637_gb300 import build as B
    d = tmp_path_factory.mktemp("waits")
    (d / "w.cu").write_text(KERNEL)
    so = str(d / "w.so")
    subprocess.run([B._nvcc()] + B.NVCC_FLAGS + ["-shared", "-I", B.CSRC, str(d / "w.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("late", [0, 1])
def test_a_copy_that_does_not_arrive_is_waited_for_twice(waits, late):
    out = (ctypes.c_ulonglong * 7)()
    assert waits.run_waits(late, ctypes.c_ulonglong(20 * MS), out) == 0
    arrived, ns, drained, drain_ns, none, none_ns, value = list(out)
    assert arrived == 0 and 20 * MS <= ns + MS < 1000 * MS  # the limit, to the timer's step
    if late:
        assert drained == 1 and value == 41
    else:
        assert drained == 0 and 20 * MS <= drain_ns + MS < 1000 * MS
    assert none == 1 and none_ns < 20 * MS
