"""The tiles of the fused FP32 step give the states of the in-place engine, bitwise.

Lattices at the edges of the dispatch: 128 x 2 and 64 x 4 tiles read by tensor
copies (rows of whole 16-byte units, at least 2^19 cells) with widths that
leave part of the last tile outside, periodic and walled; 64 x 4 tiles without
copies (odd widths); z chunks with a ragged last one; both phase-field
lattices.  The two engines share the collision and nothing of the tiles, so
the tolerance is zero.
"""
import numpy as np
import pytest

from paper_2206_11637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (nx, ny, nz, walls in all faces, h lattice)
LATTICES = [
    (128, 96, 44, True, 15),     # 128 x 2, whole tiles, walls
    (128, 97, 43, False, 15),    # ... ragged in y and z, periodic
    (256, 50, 41, False, 27),    # ... two tiles in x, D3Q27 phase field
    (236, 60, 38, True, 15),     # 128 x 2 with 20 idle columns
    (64, 130, 64, False, 15),    # 64 x 4 with copies
    (188, 61, 47, True, 27),     # ... ragged, walls
    (190, 83, 58, False, 15),    # 64 x 4 without copies: 190 x 4 bytes are no 16-byte units
    (189, 84, 59, True, 15),     # ... odd, walls
]


@pytest.mark.parametrize("nx,ny,nz,walls,lattice", LATTICES)
def test_tiles_equal_the_inplace_engine(nx, ny, nz, walls, lattice):
    from paper_2206_11637_gb300.pflbm import Simulation
    out = []
    for engine in (0, 1):
        p = W.Params(nx, ny, nz, ((1,) * 6 if walls else (0,) * 6), nu_l=0.05, gravity=(1e-6, -2e-6, 3e-6))
        p.h_lattice, p.engine = lattice, engine
        phi0 = W.sphere(p, (nx / 3.0, ny / 2.0, nz / 2.0), min(ny, nz) / 3.0)
        s = Simulation(p, phi0, W.noise((3,) + p.shape, 5, 1e-2), None, precision="fp32")
        s.step(3)
        out.append((s.time,) + s.fields() + s.populations())
        s.close()
    assert out[0][0] == out[1][0] == 3
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)
