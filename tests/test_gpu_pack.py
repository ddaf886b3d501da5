"""The copies between the dense state and the padded device layout: a state
that is set and read back is the same bit for bit, on rows that start on
16-byte boundaries and rows that do not, on buffers that are not 16-byte
aligned, and on rows longer than the copy's grid."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu


def _sim(nx, ny, precision):
    return Simulation(Config(nx=nx, ny=ny, dx=1.0, dy=1.0, dt=1e-3, s=(0.0,) * 4 + (1.0,) * 12, precision=precision))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (4, 200), (1023, 3), (1024, 5), (1026, 4), (258, 66), (5, 129), (2050, 2)])
@pytest.mark.parametrize("offset", [0, 1])
def test_set_then_get(cuda, nx, ny, precision, offset):
    import torch
    dt = torch.float32 if precision == "fp32" else torch.float64
    gen = torch.Generator(device=cuda).manual_seed(nx * 1000 + ny)
    flat = torch.rand(16 * nx * ny + offset, dtype=dt, device=cuda, generator=gen)
    f = flat[offset:].view(16, ny, nx)
    out = torch.empty(16 * nx * ny + offset, dtype=dt, device=cuda)[offset:].view(16, ny, nx)
    with _sim(nx, ny, precision) as sim:
        M.mrtlb_set_f(sim.ctx, f, True)
        M.mrtlb_get_f(sim.ctx, out, True)
        assert torch.equal(out, f)
        assert np.array_equal(sim.get_f(), f.cpu().numpy())


def test_rows_longer_than_the_grid(cuda):
    import torch
    nx = 65535 * 256 + 301
    f = torch.rand((16, 1, nx), dtype=torch.float32, device=cuda)
    with _sim(nx, 1, "fp32") as sim:
        sim.set_f(f)
        assert torch.equal(sim.get_f(on_device=True), f)
