"""The FP64 step's moments (csrc/moments.cuh) and its quotient 1.5 / rho (vquot), compiled for the host, against exact arithmetic.

Populations w (p* (1 + |u| r) + 3 c.u), r in (-1, 1): near-uniform, p* much larger than |u|.  Opposite
populations then lie within a factor of two of each other, so their differences
are exact and a first moment is off by no more than the additions of these
differences round: at most 8 of them for D3Q27, each by 2^-53 of a partial sum, which is no
larger than sum |D|.  The even moments add at most 26 values: 26 x 2^-53 x sum f.  Both hold on
every axis.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_11637_gb300", "csrc")

# the device intrinsics of the FP64 and FP32 arithmetic types as plain IEEE operations
STUB = """
#pragma once
#include <cmath>
#define __host__
#define __device__
#define __forceinline__ inline
#define R1(n, t, e) inline t n(t a) { return e; }
#define R2(n, t, o) inline t n(t a, t b) { return a o b; }
R2(__dadd_rn, double, +) R2(__dsub_rn, double, -) R2(__dmul_rn, double, *) R2(__ddiv_rn, double, /)
R2(__fadd_rn, float, +) R2(__fsub_rn, float, -) R2(__fmul_rn, float, *) R2(__fdiv_rn, float, /)
R1(__drcp_rn, double, 1 / a) R1(__frcp_rn, float, 1 / a) R1(__dsqrt_rn, double, std::sqrt(a)) R1(__fsqrt_rn, float, std::sqrt(a))
inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
"""
MAIN = """
#include "moments.cuh"
using namespace pfl;
template <int Q> void go(const double* f, double* m) {  // f by (cx+1) + 3 (cy+1) + 9 (cz+1)
  const Mom<D1> r = moments<Q, D1>([&](int cx, int cy, int cz) { return D1{f[(cx + 1) + 3 * (cy + 1) + 9 * (cz + 1)]}; });
  const D1 v[10] = {r.s, r.x, r.y, r.z, r.xx, r.yy, r.zz, r.xy, r.yz, r.xz};
  for (int k = 0; k < 10; ++k) m[k] = v[k].v;
}
extern "C" void moments_of(int q, const double* f, double* m) {
  q == 27 ? go<27>(f, m) : q == 15 ? go<15>(f, m) : go<9>(f, m);
}
extern "C" double quot(double a, double b) { return vquot(D1{a}, D1{b}, vrcp(D1{b})).v; }
"""
C27 = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]
W = {27: {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}, 15: {0: 2 / 9, 1: 1 / 9, 3: 1 / 72}, 9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("moments")
    (d / "cuda_runtime.h").write_text(STUB)
    (d / "m.cpp").write_text(MAIN)
    so = str(d / "m.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", str(d), "-I", CSRC,
                    str(d / "m.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("pstar,u", [(5.0, 1e-3), (1.0, 1e-2), (0.3, 3e-5)])
@pytest.mark.parametrize("q", [27, 15, 9])
def test_moments_of_every_axis_are_as_exact_as_their_pairs(lib, q, pstar, u):
    rng = np.random.Generator(np.random.PCG64(q))
    n2 = [sum(v * v for v in c) for c in C27]
    member = [n in W[q] and (q != 9 or c[2] == 0) for n, c in zip(n2, C27)]
    eps = Fraction(1, 2 ** 53)
    for _ in range(200):
        vel = rng.uniform(-u, u, 3)
        f = np.array([W[q][n] * (pstar * (1 + u * rng.uniform(-1, 1)) + 3 * float(np.dot(c, vel))) if m else 0.0
                      for n, c, m in zip(n2, C27, member)])
        out = np.zeros(10)
        lib.moments_of(q, f.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
        F = [Fraction(float(v)) for v in f]
        sum_d = sum(abs(F[i] - F[26 - i]) for i in range(13))
        sum_f = sum(F)
        exact = [sum(F)] + [sum(c[a] * v for c, v in zip(C27, F)) for a in range(3)]
        exact += [sum(c[a] * c[b] * v for c, v in zip(C27, F)) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))]
        for k in range(10):
            bound = 8 * eps * sum_d if 1 <= k <= 3 else 26 * eps * sum_f
            assert abs(Fraction(float(out[k])) - exact[k]) <= bound, (k, float(Fraction(float(out[k])) - exact[k]), float(bound))


def test_quotient_from_the_reciprocal_rounds_once(lib):
    """Half an ulp, and 2^-40 of one for the rounding of the correction itself."""
    lib.quot.restype = ctypes.c_double
    lib.quot.argtypes = [ctypes.c_double, ctypes.c_double]
    rng = np.random.Generator(np.random.PCG64(7))
    for rho in np.concatenate([10.0 ** rng.uniform(-4, 1, 5000), 1e-3 + rng.uniform(0, 1, 5000)]):
        got, exact = lib.quot(1.5, float(rho)), Fraction(3, 2) / Fraction(float(rho))
        ulp = Fraction(float(np.spacing(got)))
        assert abs(Fraction(got) - exact) <= ulp * (Fraction(1, 2) + Fraction(1, 2 ** 40)), rho
