"""Sides refilled before every step (walls, diffuse reflection): the
one-thread-per-node kernel works them out beside its nodes, the march reads
them from memory; both against the oracle, with such sides beside each other
and on the shortest grids that take them."""
import numpy as np
import pytest

from oracle import equilibrium as oeq
from oracle import fdlb
from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

P, O, R = ("periodic", 0, 0, 1), ("outflow", 0, 0, 1), ("reflect", 0, 0, 1)
W, W2 = ("wall", 0.1, -0.05, 1.1), ("wall", -0.1, 0.05, 0.9)
D, D2 = ("diffuse", 0.1, -0.05, 1.1), ("diffuse", -0.1, 0.05, 0.9)
SIDES = {"wall_y": (P, P, W, W2), "wall_x": (W, W2, P, P), "one_wall": (W, O, O, R), "diffuse_x": (D, D2, P, P),
         "diffuse_y": (P, P, D, D2), "wall_x_diffuse_y": (W, W2, D, D2), "wall_and_diffuse": (P, P, W, D2),
         "diffuse_corner": (D, O, R, D2)}
KERNELS = {"plain": M.MRTLB_KERNEL_PLAIN, "tiled": M.MRTLB_KERNEL_TILED}


@pytest.mark.parametrize("kernel", list(KERNELS))
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("nx,ny,version", [(3, 3, 1), (5, 34, 2), (67, 4, 3), (130, 19, 1)])
@pytest.mark.parametrize("sides", list(SIDES))
def test_steps_against_the_oracle(cuda, sides, nx, ny, version, precision, tol, kernel):
    steps = 4
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 eq_version=version, precision=precision)
    p = fdlb.Params(nx=nx, ny=ny, dx=cfg.dx, dy=cfg.dy, dt=cfg.dt, s=np.asarray(cfg.s),
                    sides=tuple(fdlb.Side(*s) for s in cfg.bc), version=version)
    f0 = fdlb.prepare(oeq.feq(*workloads.smooth_fields(nx, ny, 3), version), p)
    ref = fdlb.run(f0, p, steps)
    with Simulation(cfg) as sim:
        sim.set_kernel(KERNELS[kernel])
        sim.set_f(f0.astype(sim.fdtype))
        sim.step(steps)
        got = sim.get_f().astype(np.float64)
    # (against the state's scale: a rounding of the moments reaches every plane)
    assert np.abs(got - ref).max() / np.abs(ref).max() < tol * steps
