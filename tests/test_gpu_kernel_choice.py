"""The automatic choice between the march and the one-thread-per-node kernel,
on either side of its line: the same bits as the kernel it stands for."""
import numpy as np
import pytest

from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,precision,marches", [(700, 500, "fp32", False), (1501, 300, "fp32", True),
                                                     (1501, 701, "fp32", True), (100, 60, "fp64", False),
                                                     (200, 50, "fp64", True), (1024, 256, "fp64", True)])
def test_automatic_choice(cuda, nx, ny, precision, marches):
    cfg, fields = workloads.richtmyer_meshkov(nx=nx, ny=ny, precision=precision)
    out = {}
    for kernel in (M.MRTLB_KERNEL_AUTO, M.MRTLB_KERNEL_TILED, M.MRTLB_KERNEL_PLAIN):
        with Simulation(cfg) as sim:
            sim.set_kernel(kernel)
            sim.init_equilibrium(*fields)
            sim.step(5)
            out[kernel] = sim.get_f()
    same = M.MRTLB_KERNEL_TILED if marches else M.MRTLB_KERNEL_PLAIN
    assert np.array_equal(out[M.MRTLB_KERNEL_AUTO], out[same])
