"""The FP32 step of grids between the smallest and the march's (tiles of 32 x 4
or 16 x 8 nodes, or one thread per node where neither fits): whole and ragged
tiles, one row or column past a tile, every side without walls, against the
oracle; and the same run over a captured loop."""
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
I, I2 = ("inflow", 0.1, 0.05, 1.05, 1.1), ("inflow", -0.1, 0.0, 0.9, 0.8)
SIDES = {"periodic": (P, P, P, P), "open": (I, O, O, I2), "reflect": (R, R, R, O), "tube": (O, O, P, P)}


@pytest.mark.parametrize("nx,ny", [(64, 32), (65, 33), (63, 35), (48, 48), (49, 41), (33, 70), (20, 110), (400, 6), (2100, 1)])
@pytest.mark.parametrize("sides", list(SIDES))
@pytest.mark.parametrize("version,steps", [(1, 3), (2, 2), (3, 2), (1, 67)])
def test_steps_against_the_oracle(cuda, sides, nx, ny, version, steps):
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 eq_version=version, precision="fp32")
    p = fdlb.Params(nx=nx, ny=ny, dx=cfg.dx, dy=cfg.dy, dt=cfg.dt, s=np.asarray(cfg.s), version=version,
                    sides=tuple(fdlb.Side(*q) for q in cfg.bc))
    f0 = oeq.feq(*workloads.smooth_fields(nx, ny, 3), version)
    ref = fdlb.run(f0, p, steps)
    with Simulation(cfg) as sim:
        sim.set_kernel(M.MRTLB_KERNEL_PLAIN)
        sim.set_f(f0.astype(np.float32))
        sim.step(steps)
        got = sim.get_f().astype(np.float64)
    # (per step a few roundings of the state's scale)
    assert np.abs(got - ref).max() / np.abs(ref).max() < 2e-6 * min(steps, 10)
