"""The equilibrium of an FP32 state from FP64 fields far from order one, each
scaled by itself, on either side of the range that the arithmetic in pairs of
floats is made for: the FP64 result rounded to FP32, infinite where that is."""
import numpy as np
import pytest

from oracle import equilibrium as oeq
from paper_1106_0785_gb300 import workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("version", [1, 2])
@pytest.mark.parametrize("rho_exp", [-59, -20, 0, 20, 59])
@pytest.mark.parametrize("u_exp", [-59, -30, 0, 11, 20, 24, 26, 30, 59])
def test_magnitudes(cuda, rho_exp, u_exp, version):
    nx, ny = 67, 8
    rho, ux, uy, T = workloads.smooth_fields(nx, ny, 5)
    rho, ux, uy = rho * 2.0 ** rho_exp, ux * 2.0 ** u_exp, uy * 2.0 ** u_exp
    ux[0, 0], uy[-1, -1] = 0.0, 0.0
    cfg = Config(nx=nx, ny=ny, dx=1.0, dy=1.0, dt=1e-3, s=(0.0,) * 4 + (1.0,) * 12, eq_version=version, precision="fp32")
    with Simulation(cfg) as sim:
        for T_exp in (-59, -30, 0, 20, 40, 49, 51, 59):
            ref = oeq.feq(rho, ux, uy, T * 2.0 ** T_exp, version)
            sim.init_equilibrium(rho, ux, uy, T * 2.0 ** T_exp)
            got = sim.get_f()
            # half a last place, and the little by which 2^-40 of the largest term can
            # move a tie (or FP32's end)
            size = np.broadcast_to(np.abs(ref).max(axis=0), ref.shape)
            ends = np.abs(np.abs(ref) - 2.0 ** 128) <= 2.0 ** 104 + 2.0 ** -40 * size
            out = np.isinf(got)
            assert not np.isnan(got).any()
            assert (out == (np.abs(ref) >= 2.0 ** 128))[~ends].all() and (np.sign(got) == np.sign(ref))[out].all()
            ulp = np.spacing(np.minimum(np.abs(ref), 2.0 ** 127).astype(np.float32)).astype(np.float64)
            assert (np.abs(got[~out].astype(np.float64) - ref[~out]) <= (0.5 * ulp + 2.0 ** -40 * size)[~out]).all(), T_exp
