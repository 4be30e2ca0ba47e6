"""Forms of the fused FP32 step that lattices take beside the plain tiles: widths below the box of a
tensor copy, 64 x 4 tiles without copies on D3Q27, 64 x 4 tiles with solid cells, replays of a step
graph, and adjoint sweeps whose steps run between the live arrays, checkpoints and segment slots.
Each case names the tile it is about.

The in-place engine shares the collision and nothing of the tiles: states are compared bitwise.
With solid cells the reference is the FP64 oracle, at the bound of the smaller solid lattices
(1e-5 on phi).  The adjoint's gradient sums 10 steps of 42 populations rounded to FP32 on either
engine: 10 x 42 x 6e-8 = 2.5e-5 relative, taken as 1e-4.
"""
import os

import numpy as np
import pytest

from paper_2206_11637_gb300 import _lib as L
from paper_2206_11637_gb300 import pflbm
from paper_2206_11637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def setup(nx, ny, nz, walls, lattice, tile):
    p = W.Params(nx, ny, nz, ((1,) * 6 if walls else (0,) * 6), nu_l=0.05, gravity=(1e-6, -2e-6, 3e-6))
    p.h_lattice = lattice
    phi0 = W.sphere(p, (nx / 3.0, ny / 2.0, nz / 2.0), min(ny, nz) / 3.0)
    assert pflbm.step_tile(p, L.PFL_FP32) == tile
    return p, phi0, W.noise((3,) + p.shape, 5, 1e-2)


@pytest.mark.parametrize("nx,ny,nz,walls,lattice,tile,steps", [
    (60, 97, 91, True, 15, (64, 4, True), 3),      # rows shorter than the box, ragged
    (100, 75, 71, False, 27, (128, 2, True), 3),   # ... of 128 x 2, periodic
    (190, 83, 58, False, 27, (64, 4, False), 3),   # 64 x 4 without copies, D3Q27
    (189, 84, 59, True, 27, (64, 4, False), 3),
    (128, 97, 43, False, 15, (128, 2, True), 71),  # two replays of 32 steps and seven launches
    (64, 130, 64, True, 15, (64, 4, True), 71),
])
def test_tiles_equal_the_inplace_engine(nx, ny, nz, walls, lattice, tile, steps):
    from paper_2206_11637_gb300.pflbm import Simulation
    p, phi0, u0 = setup(nx, ny, nz, walls, lattice, tile)
    out = []
    for engine in (0, 1):
        p.engine = engine
        s = Simulation(p, phi0, u0, None, precision="fp32")
        s.step(steps)
        out.append(s.fields() + s.populations())
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("lattice", [15, 27])
def test_wide_tiles_with_solids(lattice):
    import oracle
    from paper_2206_11637_gb300.pflbm import Simulation
    p = W.Params(98, 101, 97, (0, 0, 1, 1, 0, 0), 1.0, 0.01, 0.02, 0.05, 2e-4, 0.03, 4.0, (0.0, -2e-6, 0.0))
    p.h_lattice = lattice
    x, y, z = W.coords(p)
    p.solid = ((x - 48.5) ** 2 + (z - 48.0) ** 2 > 47.0 ** 2).astype(np.uint8)
    phi0 = W.sphere(p, (48.0, 40.0, 47.0), 20.0)
    u0 = np.zeros((3,) + p.shape)
    u0[1] = -0.01 * phi0
    assert pflbm.step_tile(p, L.PFL_FP32) == (64, 4, False)
    s = Simulation(p, phi0, u0, None, precision="fp32")
    o = oracle.from_params(p, phi0, u0, None)
    s.step(12)
    o.step(12, max(1, os.cpu_count() or 1))
    fluid = p.solid == 0
    a, b = s.fields()[0], np.asarray(o.fields()[0])
    assert np.all(a[~fluid] == 0)
    assert np.abs(a[fluid] - b[fluid]).max() <= 1e-5 * np.abs(b[fluid]).max()


def test_adjoint_through_checkpoints_on_the_copy_path():
    from paper_2206_11637_gb300.pflbm import Simulation
    p, phi0, u0 = setup(128, 97, 43, False, 15, (128, 2, True))
    n, rng = 10, np.random.Generator(np.random.PCG64(3))
    # K = 4: observations at a checkpoint, inside a segment, at the last checkpoint, at the end
    obs = [(k, rng.uniform(-1, 1, p.cells) / p.cells) for k in (4, 6, 8, 10)]
    plain = Simulation(p, phi0, u0, None, precision="fp32")
    J = 0.0
    for k, w in obs:
        plain.step(k - plain.time)
        J += float(np.dot(w, plain.phi().reshape(-1)))
    got = []
    for engine in (0, 1):
        p.engine = engine
        s = Simulation(p, phi0, u0, None, precision="fp32")
        got.append(s.adjoint(n, obs))
        for a, b in zip(s.populations() + s.fields(), plain.populations() + plain.fields()):
            assert np.array_equal(a, b)
        # sums of 0.5 M products in FP64, in another order
        assert abs(got[-1][0] - J) <= 1e-12 * sum(np.abs(w).sum() for _, w in obs)
        s.close()
    (_, a), (_, b) = got
    assert np.all(np.abs(a - b) <= 1e-4 * np.abs(b))


def test_adjoint_workspace_holds_what_the_sweep_uses():
    """n = 10, K = 4: three checkpoints and K - 1 segment states, as each segment starts in its
    checkpoint; n = 1: one checkpoint alone.  Each state more costs the same."""
    from paper_2206_11637_gb300.pflbm import Simulation
    p, phi0, u0 = setup(64, 130, 64, False, 15, (64, 4, True))
    s = Simulation(p, phi0, u0, None, precision="fp32")
    state = 4 * p.cells * (15 + 27 + 1)  # of 256-byte multiples here
    size = [s.lib.pfl_adjoint_workspace_bytes(s.ctx, n) for n in (1, 2, 10, 16, 17)]
    assert [(v - size[0]) // state for v in size] == [0, 1, 5, 6, 7]  # 1+0, 1+1, 3+3, 4+3, 4+4 states
    assert all((v - size[0]) % state == 0 for v in size)
