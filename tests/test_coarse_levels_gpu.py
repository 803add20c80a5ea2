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


@pytest.mark.parametrize("nu", [(1, 1), (2, 1), (0, 2), (2, 0)])
@pytest.mark.parametrize("shape", [(32, 16, 8), (64, 32, 16)])
def test_single_block_schedules_match_the_oracle(shape, nu):
    """The coarse levels of anisotropic grids in one block, alone and below
    other levels, under every form of the schedule."""
    rho = _rough(shape, 11 * sum(shape))
    ref = O.solve(O.OracleParams(n=shape, k_max=1), rho)
    with Recon(shape, precision="mixed", k_max=1, replay_alpha=ref.alpha, nu1=nu[0], nu2=nu[1]) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.steps == 1 and st.relres[0] <= 1e-8
    assert np.linalg.norm(phi - ref.phi) <= BARS["mixed"] * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("nu", [(1, 1), (2, 1), (0, 2), (2, 0)])
@pytest.mark.parametrize("n,faces", [(32, 0), (64, 0), (64, 1)])
def test_cluster_schedules_match_the_oracle(n, faces, nu):
    """The cluster's V-cycle under every form of its schedule (no sweep before
    the restriction, none after the prolongation) and both coefficient forms,
    alone (32^3: several cycles a launch) and below a finer level."""
    rho = _rough((n, n, n), 7 * n + faces)
    ref = O.solve(O.OracleParams(n=(n, n, n), k_max=1), rho)
    with Recon((n, n, n), precision="mixed", k_max=1, replay_alpha=ref.alpha, coarse_faces=faces,
               nu1=nu[0], nu2=nu[1]) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.steps == 1 and st.relres[0] <= 1e-8
    assert np.linalg.norm(phi - ref.phi) <= BARS["mixed"] * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("s_side", [0.25, 0.2, 0.0])
@pytest.mark.parametrize("shape", [(8, 8, 32), (16, 8, 64), (8, 16, 8), (64, 64, 32)])
def test_smoothing_forms_match_the_oracle(shape, s_side):
    """S in its streaming form (pieces of a few planes up to whole columns)
    and per axis, with the default side weight and others."""
    rho = _rough(shape, sum(shape) + 1)
    ref = O.solve(O.OracleParams(n=shape, k_max=2, s_side=s_side), rho)
    with Recon(shape, k_max=2, s_side=s_side, replay_alpha=ref.alpha) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.steps == ref.steps
    assert np.linalg.norm(phi - ref.phi) <= BARS["fp64"] * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("alpha", [0.125, 0.1])
@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 8, 32), (16, 8, 64), (8, 16, 16), (32, 64, 16), (64, 32, 32)])
def test_node_displacements_match_the_oracle(shape, alpha):
    """The tracers' displacements in fixed point and in FP64 (grids that do not
    fill the tile, step lengths that are no power of two): four steps with
    every linear solve converged to rounding.  A displacement is rounded to
    2^-53 cells on one side and computed in FP64 on the other, and the fields
    after it differ by some 1e-13 (the 32^3 trajectory grows a difference less
    than tenfold in ten steps), so 1e-9 has room and catches any wrong node."""
    r = np.random.default_rng(sum(shape))
    k = np.meshgrid(*[np.arange(n) * 2 * np.pi / n for n in shape], indexing="ij")
    rho = np.exp(0.6 * np.sin(k[0] + 1) * np.cos(k[1]) + 0.5 * np.cos(k[2] + k[0]) + 0.1 * r.standard_normal(shape))
    steps = np.full(4, alpha)
    ref = O.solve(O.OracleParams(n=shape, k_max=4, tol_in=1e-13, max_vcycles=100), rho, replay_alpha=steps)
    with Recon(shape, k_max=4, tol_in=1e-13, max_vcycles=100, replay_alpha=steps) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        R.solve()
        phi, m = R.field("phi").cpu().numpy(), R.field("mass").cpu().numpy()
    assert np.linalg.norm(phi - ref.phi) <= 1e-9 * np.linalg.norm(ref.phi)
    assert np.abs(m - ref.m).max() <= 1e-9


@pytest.mark.parametrize("climiter", [0, 1, 2])
@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 8, 32), (16, 8, 64), (32, 16, 32), (32, 32, 16), (8, 16, 16)])
def test_source_and_limiter_match_the_oracle(shape, climiter):
    """The screened source and limiter on strongly deformed maps where both
    limiters act (v_m = 1.5, xi_m = 0.5), every reading of C: the step lengths
    exactly and phi within the FP64 bar."""
    r = np.random.default_rng(sum(shape) + climiter)
    k = np.meshgrid(*[np.arange(n) * 2 * np.pi / n for n in shape], indexing="ij")
    rho = np.exp(1.2 * np.sin(k[0] + 1) * np.cos(k[1]) + 0.8 * np.cos(k[2] + k[0]) + 0.3 * r.standard_normal(shape))
    kw = dict(climiter=climiter, v_m=1.5, xi_m=0.5)
    ref = O.solve(O.OracleParams(n=shape, k_max=6, tol_in=1e-12, max_vcycles=100, **kw), rho)
    with Recon(shape, k_max=6, tol_in=1e-12, max_vcycles=100, **kw) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        phi = R.field("phi").cpu().numpy()
    assert st.status == ref.status
    np.testing.assert_array_equal(st.alpha, ref.alpha)
    assert np.linalg.norm(phi - ref.phi) <= BARS["fp64"] * np.linalg.norm(ref.phi)


@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 8, 32), (64, 32, 32), (16, 64, 64), (16, 32, 16)])
def test_closing_statistics_are_those_of_the_fields(shape):
    """min det, min lambda0 and max delta_r of a solve's record are the extrema
    of the fields, to the last bit (the same FP64 arithmetic at the node that
    attains each)."""
    rho = _rough(shape, 3 * sum(shape))
    with Recon(shape, precision="mixed", k_max=5) as R:
        R.deposit_grid(torch.from_numpy(rho).cuda())
        st = R.solve()
        assert st.min_det == R.field("det").min().item()
        assert st.min_lambda0 == R.field("lambda0").min().item()
        assert st.max_delta_r == R.field("delta_r").max().item()


def test_particle_errors_leave_the_next_deposit_exact():
    """The deposit is enqueued before its inputs' checks are read back: every
    rejected catalogue (not finite, negative, without mass) reports its status
    and leaves the accumulators clear, so that the next deposit on the handle
    is that of a fresh one, bit for bit, with and without masses."""
    from paper_1611_09638_gb300 import ReconError, _abi

    n, box, count = 16, 50.0, 3001
    r = np.random.default_rng(5)
    pos = torch.from_numpy(r.uniform(-box, 2 * box, (count, 3))).cuda()
    mass = torch.from_numpy(r.uniform(0.1, 3.0, count)).cuda()

    def with_value(t, value, at):
        t = t.clone()
        t.view(-1)[at] = value
        return t

    with Recon((n, n, n), box=box) as fresh:
        fresh.deposit_particles(pos)
        unit = fresh.field("density").clone()
        fresh.deposit_particles(pos, mass)
        heavy = fresh.field("density").clone()
    assert abs(unit.sum().item() - count) <= 1e-9 * count
    assert abs(heavy.sum().item() - mass.sum().item()) <= 1e-9 * mass.sum().item()
    cases = [((with_value(pos, float("nan"), 7), None), _abi.RECON_E_NONFINITE),
             ((with_value(pos, float("inf"), 3 * count - 1), None), _abi.RECON_E_NONFINITE),
             ((with_value(pos, float("-inf"), 0), mass), _abi.RECON_E_NONFINITE),
             ((pos, with_value(mass, -1.0, 5)), _abi.RECON_E_NONFINITE),
             ((pos, with_value(mass, float("nan"), count - 1)), _abi.RECON_E_NONFINITE),
             ((pos, torch.zeros_like(mass)), _abi.RECON_E_INVALID)]
    with Recon((n, n, n), box=box) as R:
        for (p, m), status in cases:
            with pytest.raises(ReconError) as e:
                R.deposit_particles(p, m)
            assert e.value.status == status
            with pytest.raises(ReconError):
                R.field("density")
            R.deposit_particles(pos)
            assert torch.equal(R.field("density"), unit)
            R.deposit_particles(pos, mass)
            assert torch.equal(R.field("density"), heavy)
