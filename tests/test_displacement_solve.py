"""The node displacements' fixed-point solve (displacement_solve.cuh), compiled
for the host and compared with the exact rational solution."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
BITS = 53  # fraction bits of a displacement


@pytest.fixture(scope="module")
def solve_nodes(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("host") / "displacement_solve.so")
    src = os.path.join(HERE, "host", "displacement_solve.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-fPIC", "-shared",
                    "-I", os.path.join(HERE, "host"), "-o", lib, src], check=True)
    fn = ctypes.CDLL(lib).solve_nodes
    fn.restype = None

    def run(scales, h, g):
        scales, h, g = (np.ascontiguousarray(a, t) for a, t in ((scales, np.int32), (h, np.int64), (g, np.int64)))
        out, ok = np.zeros((len(h), 3), np.int64), np.zeros(len(h), np.int32)
        fn(ctypes.c_int(len(h)), *(ctypes.c_void_p(a.ctypes.data) for a in (scales, h, g, out, ok)))
        return out, ok.astype(bool)

    return run


def _exact(Q, Qd, kexp, h, g):
    """U in units of 2^-BITS cells, and the largest row sum of |e^-1|."""
    one, four = Fraction(1, 1 << Q), Fraction(1, 4 << Q)
    xx, yy, zz = (1 + int(v) * one for v in h[:3])
    xy, xz, yz = (int(v) * four for v in h[3:])
    X = [[yy * zz - yz * yz, xz * yz - xy * zz, xy * yz - yy * xz],
         [xz * yz - xy * zz, xx * zz - xz * xz, xy * xz - xx * yz],
         [xy * yz - yy * xz, xy * xz - xx * yz, xx * yy - xy * xy]]
    det = xx * X[0][0] + xy * X[0][1] + xz * X[0][2]
    G = [Fraction(int(v)) * Fraction(2) ** (BITS - 1 - Qd - kexp) for v in g]
    U = [sum(X[a][b] * G[b] for b in range(3)) / det for a in range(3)]
    return U, max(sum(abs(X[a][b]) for b in range(3)) for a in range(3)) / abs(det)


def _triads(r, count, Q):
    """Hessian sums of triads with eigenvalues in [0.2, 3]."""
    q, _ = np.linalg.qr(r.normal(size=(count, 3, 3)))
    e = np.einsum("nab,nb,ncb->nac", q, np.exp(r.uniform(np.log(0.2), np.log(3.0), (count, 3))), q)
    h = np.stack([e[:, 0, 0] - 1, e[:, 1, 1] - 1, e[:, 2, 2] - 1, 4 * e[:, 0, 1], 4 * e[:, 0, 2], 4 * e[:, 1, 2]], 1)
    return np.rint(h * 2.0 ** Q).astype(np.int64)


def _check(solve_nodes, scales, h, g):
    out, ok = solve_nodes(scales, h, g)
    assert ok.mean() >= 0.99  # (the FP64 form takes the others)
    for n in np.flatnonzero(ok):
        U, rows = _exact(*(int(v) for v in scales[n]), h[n], g[n])
        # half a unit from the final rounding, 1/8 from the pieces (they end at
        # 2^-57 cells), and the mixed entries of e, rounded to 2^-54, carried
        # through e^-1: two a row, each a quarter unit at most
        bar = Fraction(5, 8) + rows * Fraction(1, 2) * max(map(abs, U)) / (1 << BITS)
        worst = max(abs(int(out[n, a]) - U[a]) for a in range(3))
        assert worst <= bar, (n, float(worst), float(bar), g[n].tolist())


@pytest.mark.parametrize("down", [0, 8, 14, 16, 20, 28, 30, 36, 48])
def test_small_gradients_beside_a_large_bound(solve_nodes, down):
    """Nodes whose gradient is 2^-down of the largest the scale allows for: as
    exact as the others, whatever the field's maximum elsewhere."""
    r = np.random.default_rng(down)
    count, Q, Qd, kexp = 400, 54, 59, 0
    h = _triads(r, count, Q)
    # |2 G| up to 2^60 at scale 2^Qd, i.e. one cell
    g = np.rint(r.uniform(-1, 1, (count, 3)) * 2.0 ** (60 - down)).astype(np.int64)
    g[::4, 1:] = 0   # along one axis only
    g[1::4] = np.abs(g[1::4])
    _check(solve_nodes, np.tile([Q, Qd, kexp], (count, 1)), h, g)


def test_no_gradient_is_no_displacement(solve_nodes):
    h = _triads(np.random.default_rng(1), 16, 54)
    out, ok = solve_nodes(np.tile([54, 59, 3], (16, 1)), h, np.zeros((16, 3)))
    assert ok.all() and not out.any()
