"""The FP32 smallest eigenvalue that screens the closing statistics (eigen32.cuh),
compiled for the host: its error stays within the bound it returns."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lambdas(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("host") / "eigen32.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(HERE, "host"), "-o", lib,
                    os.path.join(HERE, "host", "eigen32.cpp")], check=True)
    fn = ctypes.CDLL(lib).lambdas
    fn.restype = None

    def run(h):
        lam, el = np.empty(len(h), np.float32), np.empty(len(h), np.float32)
        fn(ctypes.c_int(len(h)), *(ctypes.c_void_p(a.ctypes.data) for a in (h, lam, el)))
        return lam.astype(np.float64), el.astype(np.float64)

    return run


@pytest.mark.parametrize("low_pair", [True, False])
def test_error_is_within_its_bound(lambdas, low_pair):
    """Hessians of 1e-9 to 30, half of them with (nearly) equal two lowest (or
    highest) eigenvalues, where the closed form is worst conditioned."""
    r = np.random.default_rng(int(low_pair))
    n = 100000
    size = 10.0 ** r.uniform(-9, 1.5, (n, 1))
    gap = 10.0 ** r.uniform(-9, 0, n) * r.integers(0, 2, n)
    ev = np.stack([np.zeros(n), gap if low_pair else 1 - gap, np.ones(n)], 1) * size
    ev += r.uniform(-1, 1, (n, 1)) * size * r.integers(0, 2, (n, 1))
    q, _ = np.linalg.qr(r.normal(size=(n, 3, 3)))
    e = np.einsum("nab,nb,ncb->nac", q, ev, q)
    h = np.ascontiguousarray(np.stack([e[:, 0, 0], e[:, 1, 1], e[:, 2, 2], e[:, 0, 1], e[:, 0, 2], e[:, 1, 2]], 1),
                             np.float32)
    full = h[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].astype(np.float64).reshape(n, 3, 3)
    lam, el = lambdas(h)
    assert np.all(np.abs(lam - (1 + np.linalg.eigvalsh(full)[:, 0])) <= el)
