"""Each kernel of the adjoint step of smaller grids against the oracle's exact
tangent, at a size that takes it: 16 lanes per node, the FP64 two-pass kernels in
version 1 (blocks of one warp, and of four with a remainder) and the FP32
tiles."""
import numpy as np
import pytest
from test_gpu_adjoint import BCS, H, _adjoint, _cfg, _oracle_params, _state

from oracle import fdlb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("nx,ny,precision,tol", [(100, 21, "fp64", 1e-11), (140, 37, "fp64", 1e-11), (211, 101, "fp64", 1e-11),
                                                 (40, 23, "fp32", 1e-5), (100, 37, "fp32", 1e-5)])
def test_dot_product(cuda, nx, ny, precision, tol, bc):
    cfg = _cfg(nx, ny, BCS[bc], 1, precision)
    # (the oracle differentiates at the state that the library holds)
    f0 = _state(cfg, 100).astype(np.float32 if precision == "fp32" else np.float64).astype(np.float64)
    rng = np.random.default_rng(101)
    v, w = rng.standard_normal(f0.shape), rng.standard_normal(f0.shape)
    ds, lam0 = _adjoint(cuda, cfg, f0, 1, w=w, kernel="plain")
    Jv = fdlb.step(f0 + 1j * H * v, _oracle_params(cfg)).imag / H
    assert abs(float((w * Jv).sum()) - float((lam0 * v).sum())) < tol * np.abs(w * Jv).sum()
    for k in (4, 5, 6, 7, 9, 12, 15):
        sk = np.asarray(cfg.s, dtype=complex)
        sk[k] += 1j * H
        dF = fdlb.step(f0.astype(complex), _oracle_params(cfg, sk)).imag / H
        assert abs(ds[k] - float((w * dF).sum())) < 10 * tol * np.abs(w * dF).sum(), k
    assert np.all(ds[:4] == 0)
