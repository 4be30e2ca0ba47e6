"""The rule that picks the fused step's tile (pfl_step_tile, on the host), at its edges: width of the
rows, size, solid cells, and the launch grid's limit of 65535 blocks in y and in z, within which
lattices of many rows or planes stay."""
import pytest

from paper_2206_11637_gb300 import _lib as L
from paper_2206_11637_gb300 import build as B
from paper_2206_11637_gb300 import workloads as W
from paper_2206_11637_gb300 import pflbm

CASES = [
    # nx, ny, nz, precision, h lattice, solid, tile
    (128, 384, 128, L.PFL_FP32, 15, False, (128, 2, True)),
    (128, 384, 128, L.PFL_FP32, 15, True, (64, 4, False)),
    (128, 384, 128, L.PFL_FP16S, 15, False, (32, 8, False)),
    (128, 384, 128, L.PFL_FP64, 15, False, (32, 8, False)),
    (192, 96, 60, L.PFL_FP32, 27, False, (64, 4, True)),
    (190, 83, 58, L.PFL_FP32, 27, False, (64, 4, False)),
    (60, 100, 100, L.PFL_FP32, 15, False, (64, 4, True)),
    (200, 400, 1, L.PFL_FP32, 9, False, (32, 4, False)),
    (32, 32, 32, L.PFL_FP32, 15, False, (32, 8, False)),
    # the last and the first number of rows on either side of each tile's grid
    (128, 131070, 2, L.PFL_FP32, 15, False, (128, 2, True)),
    (128, 131071, 2, L.PFL_FP32, 15, False, (64, 4, True)),
    (128, 262140, 2, L.PFL_FP32, 15, False, (64, 4, True)),
    (128, 262141, 2, L.PFL_FP32, 15, False, (32, 8, False)),
    (190, 262140, 2, L.PFL_FP32, 15, False, (64, 4, False)),
    (190, 262141, 2, L.PFL_FP32, 15, False, (32, 8, False)),
    # ... and of planes, in chunks of 12
    (128, 1, 786420, L.PFL_FP32, 15, False, (128, 2, True)),
    (128, 1, 786421, L.PFL_FP32, 15, False, (64, 4, False)),
]


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build_library()
    return L.load()


@pytest.mark.parametrize("nx,ny,nz,precision,lattice,solid,tile", CASES)
def test_tile_of_a_lattice(nx, ny, nz, precision, lattice, solid, tile):
    p = W.Params(nx, ny, nz)
    p.h_lattice = lattice
    if solid:
        p.solid = True
    assert pflbm.step_tile(p, precision) == tile
    assert (ny + tile[1] - 1) // tile[1] <= 65535


def test_tile_of_the_inplace_engine_and_of_invalid_parameters():
    p = W.Params(128, 96, 48)
    p.engine = 1
    assert pflbm.step_tile(p, L.PFL_FP32) == (0, 0, False)
    p.nu_l = -1.0
    with pytest.raises(L.PFLError):
        pflbm.step_tile(p, L.PFL_FP32)


@pytest.mark.gpu
def test_lattice_of_many_rows_steps():
    """131136 rows of periodic sheets, beyond the grid of 128 x 2 tiles: the states of the in-place
    engine, bitwise."""
    import math
    import torch
    from paper_2206_11637_gb300.pflbm import Simulation
    out = []
    for engine in (0, 1):
        p = W.Params(128, 64 * 2049, 2, nu_l=0.05, gravity=(1e-6, -2e-6, 3e-6))
        p.engine = engine
        y = torch.arange(p.ny, dtype=torch.float64, device="cuda").view(1, p.ny, 1).expand(p.shape)
        x = torch.arange(p.nx, dtype=torch.float64, device="cuda").view(1, 1, p.nx) * (2.0 * math.pi / p.nx)
        d = (torch.remainder(y, 64.0) - 32.0).abs() - 16.0 - torch.cos(x)
        phi0 = (0.5 - 0.5 * torch.tanh(d * (2.0 / p.xi))).contiguous()
        u0 = torch.zeros((3,) + p.shape, dtype=torch.float64, device="cuda")
        u0[1] = 1e-3 * torch.sin(x + y * (2.0 * math.pi / 64.0))
        s = Simulation(p, phi0, u0, None, precision="fp32")
        s.step(3)
        f = {"phi": torch.empty(p.shape, dtype=torch.float64, device="cuda"),
             "u": torch.empty((3,) + p.shape, dtype=torch.float64, device="cuda")}
        s.fields(out=f)
        s.close()
        out.append(f)
        del s
    for k in ("phi", "u"):
        assert torch.isfinite(out[0][k]).all()
        assert torch.equal(out[0][k], out[1][k])
