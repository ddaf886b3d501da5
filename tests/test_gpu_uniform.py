"""A uniform region stays as it is, bit for bit: with the collision off (all
rates zero) every neighbour difference of the advection is an exact zero, at
every Courant number the library takes, in every step kernel."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Batch, Simulation

pytestmark = pytest.mark.gpu

KERNELS = {"plain": M.MRTLB_KERNEL_PLAIN, "tiled": M.MRTLB_KERNEL_TILED}


def _case(nx, ny, courant, precision):
    d = 1.0 / max(nx, ny)
    cfg = Config(nx=nx, ny=ny, dx=d, dy=d, dt=0.5 * courant * d, s=(0.0,) * 16, modified=False, precision=precision)
    one = np.random.default_rng(3).uniform(0.02, 0.2, (16, 1, 1))
    return cfg, np.broadcast_to(one, (16, ny, nx)).astype(np.float64 if precision == "fp64" else np.float32)


@pytest.mark.parametrize("courant", [0.1, 0.5, 0.8, 1.0])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,kernel", [(40, 30, "plain"), (200, 100, "plain"), (200, 100, "tiled"), (40, 30, "batch")])
def test_bits(cuda, nx, ny, kernel, precision, courant):
    cfg, f0 = _case(nx, ny, courant, precision)
    with Simulation(cfg) as sim:
        sim.set_f(f0)
        if kernel == "batch":
            with Batch([sim]) as b:
                b.step(100)
                b.sync()
        else:
            sim.set_kernel(KERNELS[kernel])
            sim.step(100)
        assert np.array_equal(sim.get_f(), f0)
