"""FP32 states: the equilibrium from FP64 fields and the conservation sums, both
formed on the FP32 pipe with their errors carried along, against FP64 numpy:
ordinary fields, magnitudes beyond the range that arithmetic is made for, and
values that are not finite."""
import numpy as np
import pytest

from oracle import equilibrium as oeq
from paper_1106_0785_gb300 import d2v16, workloads
from paper_1106_0785_gb300.mrtlb import Config
from paper_1106_0785_gb300.simulation import Simulation

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 70), (129, 5), (300, 200), (1030, 300)]


def _sim(nx, ny, version=1):
    return Simulation(Config(nx=nx, ny=ny, dx=1.0, dy=1.0, dt=1e-3, s=(0.0,) * 4 + (1.0,) * 12, eq_version=version,
                             precision="fp32"))


@pytest.mark.parametrize("version", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -70, 2.0 ** 70])
def test_equilibrium_is_rounded_once(cuda, nx, ny, version, scale):
    """The FP64 result rounded to FP32: half a last place, and the little by which
    2^-40 of the largest term can move a tie."""
    rho, ux, uy, T = workloads.smooth_fields(nx, ny, 5)
    rho = rho * scale
    ux[0, 0], uy[-1, -1] = 0.0, 0.0
    ref = oeq.feq(rho, ux, uy, T, version)
    with _sim(nx, ny, version) as sim:
        sim.init_equilibrium(rho, ux, uy, T)
        got = sim.get_f().astype(np.float64)
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    assert (np.abs(got - ref) <= 0.5 * ulp + 2.0 ** -40 * np.abs(ref).max(axis=0)).all()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("spread", [0, 30, 90])
def test_sums(cuda, nx, ny, spread):
    """Sums of f of one size, and of sizes 2^-spread .. 1 and above 2^60, as FP64
    has them: 2^-50 of the sum of magnitudes."""
    rng = np.random.default_rng(7)
    M = d2v16.moment_matrix()[:4]

    def state():
        f = workloads.random_distributions(nx, ny, rng.integers(1 << 30))
        f *= 2.0 ** -rng.integers(0, spread + 1, size=(1, ny, nx)) * (2.0 ** 61 if spread == 90 else 1.0)
        return f.astype(np.float32)

    f0 = state()
    with _sim(nx, ny) as sim:
        sim.set_f(f0)
        first = sim.reduce()
        sim.step(0)
        again = sim.reduce()
    terms = M[:, :, None, None] * f0.astype(np.float64)[None]
    assert (np.abs(first[:4] - terms.sum((1, 2, 3))) <= 2.0 ** -50 * np.abs(terms).sum((1, 2, 3))).all()
    assert first[4] == 0.0 and again[4] == 0.0 and np.allclose(first[:4], again[:4], rtol=1e-13, atol=0)


def test_residual(cuda):
    """max |T - T_prev| over steps, against the temperatures of the states."""
    cfg, fields = workloads.richtmyer_meshkov(nx=300, ny=70, precision="fp32")
    M = d2v16.moment_matrix()[:4]

    def temperature(f):
        rho, jx, jy, e = np.tensordot(M, f.astype(np.float64), axes=(1, 0))
        return (e * rho - 0.5 * (jx * jx + jy * jy)) / rho ** 2

    with Simulation(cfg) as sim:
        sim.init_equilibrium(*fields)
        sim.reduce()
        T0 = temperature(sim.get_f())
        sim.step(3)
        got = sim.reduce()[4]
        T1 = temperature(sim.get_f())
    ref = np.abs(T1 - T0).max()
    assert abs(got - ref) <= 2.0 ** -48 * max(T0.max(), T1.max())


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 3e38])
def test_sums_of_values_that_are_not_ordinary(cuda, bad):
    f = workloads.random_distributions(40, 30, 3).astype(np.float32)
    f[2, 7, 11] = bad
    with _sim(40, 30) as sim:
        sim.set_f(f)
        got = sim.reduce()
    with np.errstate(all="ignore"):
        rho = f.astype(np.float64).sum()
    if np.isnan(rho):
        assert np.isnan(got[0])
    elif np.isinf(rho):
        assert got[0] == rho
    else:
        assert np.isclose(got[0], rho, rtol=1e-14)
