"""The automatic kernel choice by equilibrium version and sides: on either side of
its lines the same bits as the kernel it stands for.  And the one-thread kernel
above the size at which its walls are refilled by a launch before it, against
the march."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

P, W, W2 = ("periodic", 0, 0, 1), ("wall", 0.1, -0.05, 1.1), ("wall", -0.1, 0.05, 0.9)
SIDES = {"periodic": (P, P, P, P), "walls": (P, P, W, W2)}


def _run(nx, ny, precision, version, sides, kernel, steps):
    d = 1.0 / max(nx, ny)
    cfg = Config(nx=nx, ny=ny, dx=d, dy=d, dt=0.05 * d, s=workloads.rates(800.0, 1200.0, 3000.0), bc=SIDES[sides],
                 eq_version=version, precision=precision)
    with Simulation(cfg) as sim:
        sim.set_kernel(kernel)
        sim.init_equilibrium(*workloads.smooth_fields(nx, ny, 3))
        sim.step(steps)
        return sim.get_f()


@pytest.mark.parametrize("nx,ny,precision,version,sides,marches", [
    (100, 60, "fp64", 2, "periodic", False), (100, 68, "fp64", 2, "periodic", True), (100, 72, "fp64", 1, "periodic", True),
    (49, 176, "fp64", 3, "periodic", False), (64, 170, "fp64", 3, "periodic", True), (515, 103, "fp64", 3, "periodic", False),
    (515, 103, "fp64", 1, "periodic", True), (84, 328, "fp64", 1, "periodic", False), (300, 300, "fp64", 3, "periodic", True),
    (200, 50, "fp64", 1, "walls", False), (326, 29, "fp64", 3, "walls", False), (515, 103, "fp64", 3, "walls", False),
    (256, 256, "fp64", 1, "walls", True), (1501, 300, "fp32", 3, "periodic", False), (1501, 300, "fp32", 2, "periodic", True),
    (1501, 350, "fp32", 3, "periodic", True), (1501, 280, "fp32", 1, "walls", True), (1501, 280, "fp32", 3, "walls", False)])
def test_automatic_choice(cuda, nx, ny, precision, version, sides, marches):
    same = M.MRTLB_KERNEL_TILED if marches else M.MRTLB_KERNEL_PLAIN
    auto = _run(nx, ny, precision, version, sides, M.MRTLB_KERNEL_AUTO, 5)
    assert np.array_equal(auto, _run(nx, ny, precision, version, sides, same, 5))


@pytest.mark.parametrize("nx,ny,precision,tol", [(1003, 301, "fp32", 2e-6), (1003, 303, "fp32", 2e-6), (301, 333, "fp64", 1e-12),
                                                 (301, 337, "fp64", 1e-12)])
@pytest.mark.parametrize("version", [1, 3])
def test_walls_refilled_first(cuda, nx, ny, precision, tol, version):
    steps = 4
    got = _run(nx, ny, precision, version, "walls", M.MRTLB_KERNEL_PLAIN, steps).astype(np.float64)
    ref = _run(nx, ny, precision, version, "walls", M.MRTLB_KERNEL_TILED, steps).astype(np.float64)
    # (against the state's scale: a rounding of the moments reaches every plane)
    assert np.abs(got - ref).max() / np.abs(ref).max() < tol * steps
