"""The small-grid step (one velocity per lane) at the sizes where it takes over
from the one-thread-per-node kernel, and its device table when the rates
change, against the oracle."""
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
I, W, D = ("inflow", 0.1, 0.05, 1.05, 1.1), ("wall", 0.1, -0.05, 1.1), ("diffuse", 0.1, -0.05, 1.1)
TOL = {"fp64": 1e-12, "fp32": 2e-6}


def _problem(nx, ny, bc, version, precision, modified=True, s=(800.0, 1200.0, 3000.0)):
    cfg = Config(nx=nx, ny=ny, dx=1 / 200, dy=1 / 180, dt=1e-4, s=workloads.rates(*s), bc=bc, eq_version=version,
                 modified=modified, precision=precision)
    p = fdlb.Params(nx=nx, ny=ny, dx=cfg.dx, dy=cfg.dy, dt=cfg.dt, s=np.asarray(cfg.s), version=version,
                    modified=modified, sides=tuple(fdlb.Side(*q) for q in cfg.bc))
    return cfg, p, fdlb.prepare(oeq.feq(*workloads.smooth_fields(nx, ny, 3), version), p)


# nodes: one; an odd number; one on either side of each line the choice has
@pytest.mark.parametrize("precision,nx,ny,bc", [
    ("fp64", 1, 1, (P, P, P, P)), ("fp64", 3, 5, (I, O, R, R)), ("fp64", 1000, 7, (O, I, P, P)), ("fp64", 7001, 1, (O, O, R, O)),
    ("fp64", 2000, 6, (P, P, W, W)), ("fp64", 8001, 3, (P, P, W, W)), ("fp64", 4000, 2, (P, P, D, D)),
    ("fp32", 1, 1, (P, P, P, P)), ("fp32", 400, 5, (I, O, R, R)), ("fp32", 667, 3, (O, O, P, P)),
    ("fp32", 2000, 4, (P, P, W, W)), ("fp32", 4001, 3, (P, P, W, W)), ("fp32", 2500, 4, (D, D, P, P)),
    ("fp32", 3334, 3, (P, P, D, D))])
@pytest.mark.parametrize("version,modified", [(1, True), (2, True), (3, True), (1, False)])
def test_steps_against_the_oracle(cuda, precision, nx, ny, bc, version, modified):
    steps = 3
    cfg, p, f0 = _problem(nx, ny, bc, version, precision, modified)
    ref = fdlb.run(f0, p, steps)
    with Simulation(cfg) as sim:
        sim.set_kernel(M.MRTLB_KERNEL_PLAIN)
        sim.set_f(f0.astype(sim.fdtype))
        sim.step(steps)
        got = sim.get_f().astype(np.float64)
    assert np.abs(got - ref).max() / np.abs(ref).max() < TOL[precision] * steps


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bc", [(P, P, W, W), (D, O, R, R)])
def test_new_rates(cuda, precision, bc):
    """Steps, other rates, steps, both runs long enough for the captured loop."""
    cfg, p, f0 = _problem(12, 9, bc, 1, precision)
    _, q, _ = _problem(12, 9, bc, 1, precision, s=(500.0, 900.0, 2000.0))
    ref = fdlb.run(fdlb.run(f0, p, 70), q, 70)
    with Simulation(cfg) as sim:
        sim.set_f(f0.astype(sim.fdtype))
        sim.step(70)
        sim.set_rates(q.s)
        sim.step(70)
        got = sim.get_f().astype(np.float64)
    assert np.abs(got - ref).max() / np.abs(ref).max() < TOL[precision] * 140
