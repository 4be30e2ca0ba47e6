"""FP16S states against recorded ones, bitwise.

The FP16S step rounds stochastically from a stream fixed by (cell, step), so a run
repeats itself exactly, and any change in the order of its FP32 sums shows within a few
steps as values rounded the other way.  The record (CRC-32 of the populations and
the fields after 1, 3 and 40 steps; 40 takes a graph replay) is of the collision by opposite
pairs; the fused and the in-place engine give the same states.  The inputs use
additions, products, quotients and square roots alone, which are the same on every machine.
"""
import os
import zlib

import numpy as np
import pytest

from paper_2206_11637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp16s_steps.txt")
MARKS = (1, 3, 40)

# name: (nx, ny, nz, walls, h lattice, solid cells)
CASES = {
    "plane": (70, 50, 1, (0, 0, 1, 1, 0, 0), 15, False),
    "plane_d2q9": (70, 50, 1, (0, 0, 1, 1, 0, 0), 9, False),
    "plane_solid": (70, 50, 1, (0,) * 6, 15, True),
    "box": (40, 36, 33, (1,) * 6, 15, False),
    "box_ragged_d3q27": (45, 35, 34, (0,) * 6, 27, False),
    "box_solid": (40, 36, 33, (0, 0, 1, 1, 0, 0), 15, True),
}


def inputs(name):
    nx, ny, nz, bc, lattice, solid = CASES[name]
    p = W.Params(nx, ny, nz, bc, nu_h=0.02, nu_l=0.05, sigma=1e-4, mobility=0.02, xi=5.0,
                 gravity=(1e-6, -2e-6, 0.0 if nz == 1 else 3e-6))
    p.h_lattice = lattice
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    dz = np.zeros(x.shape) if nz == 1 else z - nz / 2.0
    d = (np.sqrt((x - nx / 2.0) ** 2 + (y - ny / 2.0) ** 2 + dz ** 2) - 9.5) / 2.0
    phi0 = 0.5 - 0.5 * d / (1.0 + np.abs(d))
    n = (np.arange(3 * x.size, dtype=np.uint64) * np.uint64(2654435761)) % np.uint64(2 ** 32)
    u0 = ((n.astype(np.float64) / 2.0 ** 32 - 0.5) / 64.0).reshape((3,) + x.shape)
    if lattice == 9:
        u0[2] = 0.0
    if solid:
        p.solid = ((np.abs(x - 12) < 5) & (y < 9) | (x > nx - 4) & (y > ny // 2)).astype(np.uint8)
    return p, phi0, u0


def digests(name, engine):
    from paper_2206_11637_gb300.pflbm import Simulation
    p, phi0, u0 = inputs(name)
    p.engine = engine
    s = Simulation(p, phi0, u0, precision="fp16s")
    out = []
    for t in MARKS:
        s.step(t - s.time)
        crc = 0
        for a in s.populations() + s.fields():
            crc = zlib.crc32((np.asarray(a) + 0.0).tobytes(), crc)  # + 0.0: both zeros alike
        out.append("%08x" % crc)
    s.close()
    return out


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp16s_states_are_the_recorded_ones(name):
    with open(GOLDEN) as f:
        want = {k.split()[0]: k.split()[1:] for k in f if k.strip() and k[0] != "#"}
    for engine in (0,) if CASES[name][5] else (0, 1):
        assert digests(name, engine) == want[name], engine
