"""The FP64 reciprocal of the march and the small-grid kernels (lanes.cuh
`split_recip`: the hardware's approximation refined by two Newton-Raphson
steps) against the correctly rounded 1 / x: over all exponents its steps are
taken at, the neighbours of powers of two and the density range of the
workloads, and at zeros, infinities and NaN."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(cuda, tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("recip64") / "recip64_probe.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-o", out, os.path.join(HERE, "probes", "recip64_probe.cu")],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(out)
    lib.recip64_probe.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        r = np.empty_like(x)
        assert lib.recip64_probe(x.ctypes.data, r.ctypes.data, x.size) == 0
        return r

    return run


def _inputs():
    rng = np.random.default_rng(11)
    x = [np.ldexp(rng.uniform(1, 2, 600_000), rng.integers(-1021, 1021, 600_000)), rng.uniform(0.05, 20.0, 400_000)]
    p2 = np.ldexp(1.0, np.arange(-1020, 1021, 8))
    x.append((p2.view(np.int64)[:, None] + np.arange(-32, 33)[None, :]).ravel().view(np.float64))
    x = np.concatenate(x)
    return np.concatenate([x, -x[::7]])


def test_within_one_ulp_of_the_correctly_rounded_reciprocal(probe):
    x = _inputs()
    got, exact = probe(x), 1.0 / x
    ulps = np.abs(got.view(np.int64) - exact.view(np.int64))
    assert ulps.max() <= 1, x[np.argmax(ulps)]


def test_ends_of_the_range(probe):
    got = probe([0.0, -0.0, np.inf, -np.inf, np.nan])
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[4])
    assert got[2] == 0.0 and got[3] == 0.0 and not np.signbit(got[2]) and np.signbit(got[3])
    # beyond the steps' range: no NaN, and never on the other side of 1 / x's end
    small, large = probe(np.ldexp(1.5, [-1074, -1060, -1023])), probe(np.ldexp(1.5, [1022, 1023]))
    assert (small >= 2.0 ** 1000).all() and (large >= 0.0).all() and (large <= 2.0 ** -1000).all()
