"""The FP32 adjoint step in tiles (grids above the smallest, and versions 2 and
3 on any) against the fused march, which forms the same transposes: tiles of
32 x 4, 16 x 8 and 8 x 16 nodes, whole and ragged, one row or column past a
tile, grids of a few nodes, every kind of side, with and without the rate
gradients."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

P, O, R = ("periodic", 0, 0, 1), ("outflow", 0, 0, 1), ("reflect", 0, 0, 1)
I, W, W2 = ("inflow", 0.1, 0.05, 1.05, 1.1), ("wall", 0.1, -0.05, 1.1), ("wall", -0.1, 0.05, 0.9)
D, D2 = ("diffuse", 0.1, -0.05, 1.1), ("diffuse", -0.1, 0.05, 0.9)
SIDES = {"periodic": (P, P, P, P), "walls_x": (W, W2, P, P), "open": (I, O, W, R), "diffuse": (D, D2, R, O)}


# FP32 rounding over two steps, summed in another order: 2e-5 of the largest
# gradient, and twenty times that of the rates' (sums of terms that cancel).
@pytest.mark.parametrize("version,nx,ny", [(1, 94, 130), (1, 95, 131), (1, 14, 862), (1, 1502, 8), (1, 6, 2001), (1, 350, 37),
                                           (2, 3, 3), (2, 30, 2), (3, 31, 15), (2, 33, 70), (3, 62, 34)])
@pytest.mark.parametrize("sides", list(SIDES))
@pytest.mark.parametrize("modified", [True, False])
def test_gradients(cuda, sides, version, nx, ny, modified):
    import torch
    if ny < 3 and sides == "open":
        pytest.skip("a wall needs a fluid row beside it and one beyond")
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 eq_version=version, modified=modified, precision="fp32")
    fields = workloads.smooth_fields(nx, ny, 3)
    seed = torch.from_numpy(np.random.default_rng(nx).standard_normal((4, ny, nx))).to(cuda)
    out = {}
    for kernel in (M.MRTLB_KERNEL_AUTO, M.MRTLB_KERNEL_TILED):
        with Simulation(cfg) as sim:
            sim.set_kernel(kernel)
            sim.init_equilibrium(*fields)
            sim.adjoint_forward(2)
            ds, df = sim.adjoint_backward(dL_dmacros=seed)
            _, df_only = sim.adjoint_backward(dL_dmacros=seed, want_ds=False)
            out[kernel] = ds, df.cpu().numpy(), df_only.cpu().numpy()
    (ds, df, df_only), (ds2, df2, _) = out[M.MRTLB_KERNEL_AUTO], out[M.MRTLB_KERNEL_TILED]
    assert np.abs(df - df2).max() <= 2e-5 * np.abs(df2).max()
    assert np.abs(df_only - df2).max() <= 2e-5 * np.abs(df2).max()
    if modified:  # (without it a state that starts at equilibrium has rounding errors for m - m^eq)
        assert np.abs(ds - ds2).max() <= 20 * 2e-5 * np.abs(ds2).max()
