"""Gradients of a run on a context that a run before it left full of NaN: the
ghosts that no advanced node reads (beside wall nodes) still hold them, and
lambda must not.  Every adjoint kernel, against a fresh context."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.mrtlb import Config, MrtlbError
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

P, W, W2, D = ("periodic", 0, 0, 1), ("wall", 0.1, 0.0, 1.1), ("wall", -0.1, 0.0, 0.9), ("diffuse", 0.05, 0.0, 1.0)
SIDES = {"wall_y": (P, P, W, W2), "wall_x": (W, W2, P, P), "wall_x_diffuse_y": (W, W2, D, D)}


def _gradients(sim, fields, seed):
    sim.init_equilibrium(*fields)
    sim.adjoint_forward(6, interval=3)  # (the second segment starts in the context's second buffer)
    ds, df0 = sim.adjoint_backward(seed)
    return ds, df0.cpu().numpy()


@pytest.mark.parametrize("sides", list(SIDES))
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("version", [1, 3])
@pytest.mark.parametrize("nx,ny,kernel", [(20, 30, M.MRTLB_KERNEL_PLAIN), (100, 61, M.MRTLB_KERNEL_PLAIN),
                                          (100, 61, M.MRTLB_KERNEL_TILED)])
def test_after_a_run_that_blew_up(cuda, nx, ny, kernel, version, precision, sides):
    import torch
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 eq_version=version, precision=precision)
    fields = workloads.smooth_fields(nx, ny, 3)
    seed = torch.ones((4, ny, nx), dtype=torch.float64, device="cuda")
    with Simulation(cfg) as sim:
        sim.set_kernel(kernel)
        ds, df0 = _gradients(sim, fields, seed)
    with Simulation(cfg) as sim:
        sim.set_kernel(kernel)
        sim.set_f(np.full((16, ny, nx), np.nan))
        sim.adjoint_forward(1, interval=1)
        with pytest.raises(MrtlbError):
            sim.adjoint_backward(seed)
        ds2, df02 = _gradients(sim, fields, seed)
    assert np.isfinite(df0).all() and np.array_equal(df02, df0)
    # (sums of the rates by atomics: their order may differ)
    assert np.allclose(ds2, ds, rtol=1e-9, atol=1e-12 * np.abs(ds).max())
