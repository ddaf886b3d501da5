"""The adjoint step on 16 lanes per node (small grids, version 1) against the
fused march, which forms the same transposes a thread per node: the gradient by
the initial state and by the rates over two steps, for every kind of side and
pairs of them, grids of a few nodes, and either side of the line at which the
two-pass kernels take over."""
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
SIDES = {"periodic": (P, P, P, P), "walls_y": (P, P, W, W2), "walls_x": (W, W2, P, P), "one_wall": (I, O, W, R),
         "diffuse": (D, D2, R, R), "open": (I, O, O, R), "walls_diffuse": (W, W2, D, D2)}


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 5), (33, 7), (57, 70), (64, 63), (81, 74), (100, 61)])
@pytest.mark.parametrize("sides", list(SIDES))
@pytest.mark.parametrize("modified", [True, False])
def test_gradients(cuda, sides, nx, ny, precision, tol, modified):
    import torch
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 modified=modified, precision=precision)
    fields = workloads.smooth_fields(nx, ny, 3)
    rng = np.random.default_rng(nx)
    seed = torch.from_numpy(rng.standard_normal((4, ny, nx))).to(cuda)
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
    assert np.abs(df - df2).max() <= tol * np.abs(df2).max()
    assert np.abs(df_only - df2).max() <= tol * np.abs(df2).max()
    # Each rate's gradient is a sum over nodes of terms that largely cancel.
    # (Without the modification a state that starts at equilibrium has none:
    # m - m^eq is a rounding error at every node.)
    if modified:
        assert np.abs(ds - ds2).max() <= 20 * tol * np.abs(ds2).max()
