"""Grids that no streaming tile fits (a last axis of 8, or of 16 with a middle
axis of 8): the step limiter and the displacements a thread a node, against the
oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1611_09638_gb300 import Recon

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(16, 32, 8), (32, 8, 16), (64, 64, 8)]


def _density(shape, noise):
    r = np.random.default_rng(sum(shape))
    k = np.meshgrid(*[np.arange(n) * 2 * np.pi / n for n in shape], indexing="ij")
    return np.exp(1.2 * np.sin(k[0] + 1) * np.cos(k[1]) + 0.8 * np.cos(k[2] + k[0]) + noise * r.standard_normal(shape))


@pytest.mark.parametrize("shape", SHAPES)
def test_limiter_takes_the_oracles_steps(shape):
    """Strongly deformed maps: every step length exactly."""
    rho = _density(shape, 0.3)
    kw = dict(v_m=1.5, xi_m=0.5)
    ref = O.solve(O.OracleParams(n=shape, k_max=6, tol_in=1e-12, max_vcycles=100, **kw), rho)
    with Recon(shape, k_max=6, tol_in=1e-12, max_vcycles=100, **kw) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.status == ref.status
    np.testing.assert_array_equal(st.alpha, ref.alpha)
    assert np.linalg.norm(phi - ref.phi) <= 1e-6 * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("alpha", [0.125, 0.1])
@pytest.mark.parametrize("shape", SHAPES)
def test_displacements(shape, alpha):
    """In fixed point, and in FP64 (a step length that is no power of two): four
    steps with every linear solve converged to rounding.  A displacement is
    within some units of 2^-53 cells on both sides and the fields after it within
    1e-13, which four steps grow less than tenfold; 1e-9 has room and catches any
    wrong node."""
    rho = _density(shape, 0.1) ** 0.5
    steps = np.full(4, alpha)
    ref = O.solve(O.OracleParams(n=shape, k_max=4, tol_in=1e-13, max_vcycles=100), rho, replay_alpha=steps)
    with Recon(shape, k_max=4, tol_in=1e-13, max_vcycles=100, replay_alpha=steps) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        R.solve()
        phi, m = R.field("phi").cpu().numpy(), R.field("mass").cpu().numpy()
    assert np.linalg.norm(phi - ref.phi) <= 1e-9 * np.linalg.norm(ref.phi)
    assert np.abs(m - ref.m).max() <= 1e-9
