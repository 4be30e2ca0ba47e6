"""The waits of the tensor-copy step: a copy that does not arrive ends a wait at its limit, the
block waits once more for the same copy before it leaves, and the library reports the state as
lost until it is replaced.

The waits (csrc/tma.cuh) run in a kernel of their own, whose copy is withheld, or issued only
after the first wait has run out; no copy is in flight when a block that gave up ends.  In the library
the report word is set from the host.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2206_11637_gb300 import _lib as L
from paper_2206_11637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KERNEL = r"""
#include "tma.cuh"
using namespace pfl;
// res: first wait, its ns, second wait, its ns, wait at a barrier without copies, its ns, the value copied
__global__ void k_waits(const int* src, int late, unsigned limit, unsigned* res) {
  __shared__ unsigned long long mbar[2];
  __shared__ __align__(16) int dst[4];
  const unsigned a = smem_u32(mbar), b = smem_u32(mbar + 1);
  if (threadIdx.x == 0) {
    mbar_init(a);
    mbar_init(b);
    mbar_expect(a, 16);
  }
  __syncthreads();
  const unsigned t0 = timer_ns();
  const bool w = copy_wait(a, 0, limit);
  const unsigned t1 = timer_ns();
  __syncthreads();
  if (late && threadIdx.x == 0)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], 16, [%2];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(a) : "memory");
  const unsigned t2 = timer_ns();
  const bool d = copy_wait(a, 0, limit);
  const unsigned t3 = timer_ns();
  const bool e = copy_wait(b, -1, limit);
  const unsigned t4 = timer_ns();
  if (threadIdx.x == 0) {
    const unsigned v[7] = {w, t1 - t0, d, t3 - t2, e, t4 - t3, d ? (unsigned)dst[0] : 0};
    for (int k = 0; k < 7; ++k) res[k] = v[k];
  }
}
extern "C" int run_waits(int late, unsigned limit, unsigned* out) {
  int *src, one[4] = {41, 0, 0, 0};
  unsigned* res;
  if (cudaMalloc(&src, 16) != cudaSuccess || cudaMalloc(&res, 28) != cudaSuccess) return 1;
  cudaMemcpy(src, one, 16, cudaMemcpyHostToDevice);
  k_waits<<<1, 64>>>(src, late, limit, res);
  const cudaError_t e = cudaMemcpy(out, res, 28, cudaMemcpyDeviceToHost);
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
    out = (ctypes.c_uint * 7)()
    assert waits.run_waits(late, ctypes.c_uint(20 * MS), out) == 0
    arrived, ns, drained, drain_ns, none, none_ns, value = list(out)
    assert arrived == 0 and 20 * MS <= ns + MS < 1000 * MS  # the limit, to the timer's step
    if late:
        assert drained == 1 and value == 41
    else:
        assert drained == 0 and 20 * MS <= drain_ns + MS < 1000 * MS
    assert none == 1 and none_ns < 20 * MS


def test_a_lost_copy_is_reported_until_the_state_is_replaced():
    from paper_2206_11637_gb300.pflbm import Simulation
    p = W.Params(128, 96, 44, (1,) * 6, nu_l=0.05)  # tensor copies
    phi0, u0 = W.sphere(p, (60, 48, 22), 15), W.noise((3,) + p.shape, 5, 1e-2)
    s, ref = (Simulation(p, phi0, u0, precision="fp32") for _ in range(2))
    s.step(2)
    ref.step(2)
    h, g = s.populations()
    saved = s.save()
    for replace in (lambda: s.set_populations(h, g), lambda: s.load(saved)):
        s.workspace[-128:].view(dtype=s.torch.int32)[0] = 1  # the report word, in the last 256 bytes
        for call in (lambda: s.step(3), lambda: s.step(40)):  # launches, and a graph replay
            call()
            for read in (s.fields, s.populations, s.save, s.max_speed, s.diag, lambda: s.interface_height(0, 0)):
                with pytest.raises(L.PFLError) as e:
                    read()
                assert e.value.status == L.PFL_ERR_CUDA and "did not arrive" in str(e.value)
        replace()
        s.fields()
    assert s.time == ref.time == 2
    s.step(40)
    ref.step(40)
    for a, b in zip(s.populations() + s.fields(), ref.populations() + ref.fields()):
        assert np.array_equal(a, b)
