"""Walls in FP32 lose or gain nothing on average: the equilibrium of the side and
that of the node beside it are subtracted as moments, at the size of their
difference, so over many nodes the rounding of the wall's density and that of
the step beside it average out.  (The sides' constants are exact in FP32 here.)
A difference of two full states has a rounding of its own sign at every node,
1e-7 of the wall's density and 2e-8 of a step."""
import numpy as np
import pytest

from oracle import equilibrium as oeq
from oracle import fdlb
from paper_1106_0785_gb300 import d2v16, workloads
from paper_1106_0785_gb300 import mrtlb as M
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

P, W, W2 = ("periodic", 0, 0, 1), ("wall", 0.125, 0.0, 1.0), ("wall", -0.125, 0.0, 1.0)


@pytest.mark.parametrize("n,across,kernel", [(1000, 4, M.MRTLB_KERNEL_PLAIN), (1000, 12, M.MRTLB_KERNEL_PLAIN),
                                             (1000, 12, M.MRTLB_KERNEL_TILED)])
@pytest.mark.parametrize("axis", ["x", "y"])
def test_mean_of_many_walls(cuda, axis, n, across, kernel):
    nx, ny = (n, across) if axis == "y" else (across, n)
    bc = (P, P, W, W2) if axis == "y" else tuple((k, uy, ux, T) for k, ux, uy, T in (W, W2)) + (P, P)
    d = 1 / 200
    cfg = Config(nx=nx, ny=ny, dx=d, dy=d, dt=0.5 * d, s=workloads.rates(20.0, 30.0, 50.0), bc=bc, precision="fp32")
    p = fdlb.Params(nx=nx, ny=ny, dx=d, dy=d, dt=cfg.dt, s=np.asarray(cfg.s), sides=tuple(fdlb.Side(*s) for s in bc))
    conserved = d2v16.moment_matrix()[:4]

    def rows(f, first):  # the conserved moments on the rows `first` from either side
        m = np.tensordot(conserved, f, axes=(1, 0))
        if axis == "x":
            m = m.transpose(0, 2, 1)
        return m[:, [first, -1 - first]]

    walls, steps = [], []
    with Simulation(cfg) as sim:
        sim.set_kernel(kernel)
        for seed in range(10):
            f0 = fdlb.prepare(oeq.feq(*workloads.smooth_fields(nx, ny, seed, modes=5)), p).astype(np.float32)
            sim.set_f(f0)
            ref = fdlb.prepare(f0.astype(np.float64), p)
            walls.append(rows(sim.get_f().astype(np.float64) - ref, 0))
            sim.step(1)
            steps.append(rows(sim.get_f().astype(np.float64) - fdlb.run(ref, p, 1), 1))
    mean = np.concatenate(walls, axis=2).mean(axis=2)  # [moment][side]
    assert np.abs(mean[0]).max() <= 2.0 ** -26
    mean = np.concatenate(steps, axis=2).mean(axis=2)
    assert np.abs(mean[:3]).max() <= 2.0 ** -27  # (density and momentum)
