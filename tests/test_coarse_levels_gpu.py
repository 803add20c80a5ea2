"""The coarse end of the V-cycle against the oracle on the shapes where its
kernels change: the smallest grids (the 4^3 level right below the finest one),
anisotropic hierarchies (spacing factors that differ per axis on the 4^3
level), and the cluster's own 32^3 level at the top and below others.

Bars: phi relative L2 <= 1e-6 in FP64 and <= 1e-4 in mixed precision, the
method's stated tolerances, on the oracle's own step lengths.
"""
import numpy as np
import pytest

import oracle as O
from paper_1611_09638_gb300 import Recon

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BARS = {"fp64": 1e-6, "mixed": 1e-4}


def _rough(shape, seed):
    """A density with strong cell-to-cell contrast and empty cells."""
    r = np.random.default_rng(seed)
    rho = np.exp(1.2 * r.standard_normal(shape))
    rho[r.random(shape) < 0.05] = 0.0
    return np.ascontiguousarray(rho)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 16, 32), (64, 8, 8), (16, 16, 16), (32, 32, 32), (64, 64, 64)])
def test_coarse_levels_match_the_oracle(shape, precision):
    rho = _rough(shape, sum(shape))
    ref = O.solve(O.OracleParams(n=shape, k_max=2), rho)
    with Recon(shape, precision=precision, k_max=2, replay_alpha=ref.alpha) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.steps == ref.steps
    assert np.linalg.norm(phi - ref.phi) <= BARS[precision] * np.linalg.norm(ref.phi)
