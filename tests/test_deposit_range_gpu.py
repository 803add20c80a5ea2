"""The particle deposit at the ends of its range: the longest axes and positions
far outside the box, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1611_09638_gb300 import Recon

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(4096, 8, 8), (8, 4096, 8), (8, 8, 4096), (2048, 16, 8), (8, 16, 1024)])
def test_positions_along_the_longest_axes(shape):
    """Particles over the whole of every axis (past 2^11 cells on one of 4096
    nodes), on nodes, and up to two thousand boxes outside, where they are
    wrapped.  Cells of unit size and positions in multiples of 2^-20, so that
    no rounding comes before the deposit.  20001 unit masses have a fixed-point
    unit of 2^-46, and the three splits of a mass move a corner's charge by at
    most 1.5 of it; the oracle's roundings (2^-53 of a charge, 2^-50 a sum) are
    covered by the other half unit.  A cell takes charges from the particles of
    eight cells."""
    r = np.random.default_rng(sum(shape))
    count = 20001
    pos = np.rint(r.uniform(0, 1, (count, 3)) * shape * 2.0 ** 20) / 2.0 ** 20
    pos[::5] = np.floor(pos[::5])
    pos[1::5] += np.asarray(shape) * r.integers(-2000, 2001, (len(pos[1::5]), 3))
    pos[2::5] += np.asarray(shape) * r.integers(-1, 2, (len(pos[2::5]), 3))
    ref = O.cic_deposit(shape, pos)
    home = np.ravel_multi_index(np.floor(pos).astype(np.int64).T % np.asarray(shape)[:, None], shape)
    charges = 8 * np.bincount(home).max()
    with Recon(shape) as R:
        R.deposit_particles(torch.from_numpy(pos).cuda())
        rho = R.field("density").cpu().numpy()
    assert np.abs(rho - ref).max() <= 2 * charges * 2.0 ** -46


@pytest.mark.parametrize("exponent", [900, 985, 1000, 1009])
def test_masses_up_to_the_end_of_the_range(exponent):
    """The fixed point's unit follows the total mass by powers of two, so masses
    times 2^exponent (a total of up to 2^1023) give the density times that, bit
    for bit."""
    r = np.random.default_rng(exponent)
    pos = torch.from_numpy(r.uniform(0, 16, (5000, 3))).cuda()
    mass = torch.from_numpy(r.uniform(0.5, 1.5, 5000)).cuda()
    with Recon((16, 16, 16)) as R:
        R.deposit_particles(pos, mass)
        rho = R.field("density").clone()
        R.deposit_particles(pos, mass * 2.0 ** exponent)
        assert torch.equal(R.field("density"), rho * 2.0 ** exponent)
