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
def host(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("host") / "displacement_solve.so")
    src = os.path.join(HERE, "host", "displacement_solve.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-fPIC", "-shared",
                    "-I", os.path.join(HERE, "host"), "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


@pytest.fixture(scope="module")
def solve_nodes(host):
    fn = host.solve_nodes
    fn.restype = None

    def run(scales, h, g):
        scales, h, g = (np.ascontiguousarray(a, t) for a, t in ((scales, np.int32), (h, np.int64), (g, np.int64)))
        out, ok = np.zeros((len(h), 3), np.int64), np.zeros(len(h), np.int32)
        fn(ctypes.c_int(len(h)), *(_ptr(a) for a in (scales, h, g, out, ok)))
        return out, ok.astype(bool)

    return run


PHI_BITS = 54


def _exact(Qd, kexp, h, g):
    """U in units of 2^-BITS cells, and the largest row sum of |e^-1|."""
    one, four = Fraction(1, 1 << PHI_BITS), Fraction(1, 4 << PHI_BITS)
    G = [Fraction(int(v)) * Fraction(2) ** (BITS - 1 - Qd - kexp) for v in g]
    return _solution([1 + int(v) * one for v in h[:3]] + [int(v) * four for v in h[3:]], G)


def _solution(e, G):
    xx, yy, zz, xy, xz, yz = e
    X = [[yy * zz - yz * yz, xz * yz - xy * zz, xy * yz - yy * xz],
         [xz * yz - xy * zz, xx * zz - xz * xz, xy * xz - xx * yz],
         [xy * yz - yy * xz, xy * xz - xx * yz, xx * yy - xy * xy]]
    det = xx * X[0][0] + xy * X[0][1] + xz * X[0][2]
    U = [sum(X[a][b] * G[b] for b in range(3)) / det for a in range(3)]
    return U, max(sum(abs(X[a][b]) for b in range(3)) for a in range(3)) / abs(det)


def _triads(r, count):
    """Hessian sums of triads with eigenvalues in [0.2, 3]."""
    q, _ = np.linalg.qr(r.normal(size=(count, 3, 3)))
    e = np.einsum("nab,nb,ncb->nac", q, np.exp(r.uniform(np.log(0.2), np.log(3.0), (count, 3))), q)
    h = np.stack([e[:, 0, 0] - 1, e[:, 1, 1] - 1, e[:, 2, 2] - 1, 4 * e[:, 0, 1], 4 * e[:, 0, 2], 4 * e[:, 1, 2]], 1)
    return np.rint(h * 2.0 ** PHI_BITS).astype(np.int64)


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
    count, Qd, kexp = 400, 59, 0
    h = _triads(r, count)
    # |2 G| up to 2^60 at scale 2^Qd, i.e. one cell
    g = np.rint(r.uniform(-1, 1, (count, 3)) * 2.0 ** (60 - down)).astype(np.int64)
    g[::4, 1:] = 0   # along one axis only
    g[1::4] = np.abs(g[1::4])
    _check(solve_nodes, np.tile([Qd, kexp], (count, 1)), h, g)


def test_no_gradient_is_no_displacement(solve_nodes):
    h = _triads(np.random.default_rng(1), 16)
    out, ok = solve_nodes(np.tile([59, 3], (16, 1)), h, np.zeros((16, 3)))
    assert ok.all() and not out.any()


@pytest.mark.parametrize("Q", [54, 61, 120])
def test_values_of_any_size_modulo_2_64(host, Q):
    r = np.random.default_rng(Q)
    x = np.ldexp(r.uniform(-1, 1, 4000), r.integers(-140, 80, 4000))
    x[:6] = 0.0, -0.0, 1023.999, -1024.0, 2.0 ** -Q, 1.5 * 2.0 ** -Q
    got = np.zeros(len(x), np.uint64)
    host.fixed_mod(ctypes.c_int(len(x)), _ptr(x), ctypes.c_int(Q), _ptr(got))
    for v, w in zip(x, got):
        m = abs(Fraction(float(v))) * (1 << Q)
        n = (2 * m.numerator + m.denominator) // (2 * m.denominator)  # to nearest, halves away from 0
        assert int(w) == (n if v > 0 else -n) % (1 << 64), v


@pytest.mark.parametrize("offset", [0.0, 3.0, 60.0, 382.0, 5000.0, 2.0e5])
def test_nodes_of_a_large_potential(host, offset):
    """A node from its FP64 values: as exact where phi (and dphi) is hundreds of
    cells elsewhere, or at the node itself, as where it is small."""
    r = np.random.default_rng(int(offset))
    count, alpha = 300, 0.25
    x = np.stack(np.meshgrid(*[np.arange(-1, 2)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(float)

    def quadratics(diagonal, slope):  # 27 values each, with FP64 roundings of their own
        a = r.uniform(-1, 1, (count, 3, 3)) * 0.3
        a = a + a.transpose(0, 2, 1) + diagonal * np.eye(3)
        return (0.5 * np.einsum("pa,nab,pb->np", x, a, x) + slope * (r.uniform(-1, 1, (count, 3)) @ x.T)
                + offset * r.uniform(0.5, 1.0, (count, 1)))

    phi, dphi = quadratics(0.2, 4.0), quadratics(0.0, 1.0)
    out, ok = np.zeros((count, 3), np.int64), np.zeros(count, np.int32)
    host.displace_nodes(ctypes.c_int(count), ctypes.c_double(alpha), ctypes.c_double(1.7), ctypes.c_double(offset),
                        ctypes.c_int(0), _ptr(phi), _ptr(dphi), _ptr(out), _ptr(ok))
    assert ok.mean() >= 0.9
    for n in np.flatnonzero(ok):
        f, w = ([[[Fraction(float(v)) for v in row] for row in plane] for plane in a[n].reshape(3, 3, 3)]
                for a in (phi, dphi))
        c = 2 * f[1][1][1]
        quarter = Fraction(1, 4)
        e = [1 + f[2][1][1] - c + f[0][1][1], 1 + f[1][2][1] - c + f[1][0][1], 1 + f[1][1][2] - c + f[1][1][0],
             quarter * (f[2][2][1] - f[2][0][1] - f[0][2][1] + f[0][0][1]),
             quarter * (f[2][1][2] - f[2][1][0] - f[0][1][2] + f[0][1][0]),
             quarter * (f[1][2][2] - f[1][2][0] - f[1][0][2] + f[1][0][0])]
        unit = Fraction(alpha) / 2 * (1 << BITS)
        G = [unit * (w[2][1][1] - w[0][1][1]), unit * (w[1][2][1] - w[1][0][1]), unit * (w[1][1][2] - w[1][1][0])]
        U, rows = _solution(e, G)
        # as above (5/8), and phi's own rounding to 2^-54: a diagonal entry of e
        # moves by two units of 2^-54 at most, a mixed one by one (its rounding
        # to 2^-54 among them), so a row by four, i.e. 2 units of 2^-53; dphi's
        # (2^-60 here, alpha below 1) by less than 1/64
        bar = Fraction(5, 8) + rows * (2 * max(map(abs, U)) / (1 << BITS) + Fraction(1, 64))
        worst = max(abs(int(out[n, a]) - U[a]) for a in range(3))
        assert worst <= bar, (n, float(worst), float(bar))


def test_when_the_fixed_point_form_is_off(host):
    phi = np.zeros((1, 27))
    dphi = np.arange(27.0)[None] * 0.01
    out, ok = np.zeros((1, 3), np.int64), np.zeros(1, np.int32)

    def accepted(alpha=0.5, max_g=0.1, sum_dphi=0.0, wide=0):
        host.displace_nodes(ctypes.c_int(1), ctypes.c_double(alpha), ctypes.c_double(max_g),
                            ctypes.c_double(sum_dphi), ctypes.c_int(wide), _ptr(phi), _ptr(dphi), _ptr(out), _ptr(ok))
        return bool(ok[0])

    assert accepted() and accepted(alpha=1.0) and accepted(alpha=2.0 ** -40)
    for alpha in (0.1, 2.0, 0.0, -0.5, 2.0 ** -41, float("inf"), float("nan")):
        assert not accepted(alpha=alpha)
    for value in (float("inf"), float("nan")):
        assert not accepted(max_g=value) and not accepted(sum_dphi=value)
    assert not accepted(max_g=2.0 ** 91) and not accepted(wide=1)
