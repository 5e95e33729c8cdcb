"""DMD extrapolation evaluates its candidates in a batch whose spare instances are masked: the same
result whatever batch is left from an earlier call, no cost for the spare ones, and the convergence
masks of a run stay as they are."""
import time

import numpy as np
import pytest

import pcf_inputs as gi
from oracle import PCFOracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as m
    m.load_library()
    return m


def _snapshots(grid, directions, M, seed=0):
    o = PCFOracle(*grid)
    rng = np.random.default_rng(seed)
    star = o.to_psi(gi.random_perturbation(*grid, 0.05, seed + 1))
    Q, _ = np.linalg.qr(rng.standard_normal((o.psi_dim(), directions)))
    a, mu = 0.01 * rng.standard_normal(directions), np.linspace(0.5, 0.95, directions)
    return torch.from_numpy(np.stack([star + Q @ (a * mu ** k) for k in range(M + 1)])).cuda()


@pytest.mark.parametrize("batch,precision", [(1, 0), (3, 0), (6, 0), (1, 1)])
def test_result_does_not_depend_on_the_evaluation_batch(pcf, batch, precision):
    """A low-rank call alone, and after a call of many candidates has made a larger batch."""
    grid = (16, 17, 16)
    low, high = _snapshots(grid, 1, 8), _snapshots(grid, 7, 20, 3)
    s = pcf.Solver(*grid, batch=batch, precision=precision, solve_kind=2 if precision else 0)
    u, r, J = s.dmd_extrapolate(low, rank_tol=1e-10)
    u = u.clone()
    s.dmd_extrapolate(high, rank_tol=1e-10)
    v, r2, J2 = s.dmd_extrapolate(low, rank_tol=1e-10)
    assert r2 == r and J2 == J and torch.equal(u, v)
    s.close()


def test_low_rank_costs_less_than_full_rank(pcf):
    """Two candidates of 64 x 65 x 64 take well under the time of twenty; with every spare instance
    evaluated as well both took about that."""
    grid = (64, 65, 64)
    s, times = pcf.Solver(*grid), []
    low = _snapshots(grid, 1, 20)
    noise = torch.randn(low.shape, dtype=low.dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    for S in (low + 1e-3 * low.abs() * noise, low):
        best = np.inf
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            s.dmd_extrapolate(S, rank_tol=1e-10)
            best = min(best, time.perf_counter() - t)
        times.append(best)
    assert times[1] <= 0.6 * times[0]


def test_a_jump_keeps_the_masks_of_the_run(pcf):
    """An instance that has converged stays as it is while the others jump."""
    grid = (16, 17, 16)
    us = gi.batch(gi.random_perturbation, range(6), *grid, 0.1)
    us[0] *= 1e-12
    o = PCFOracle(*grid)
    hist = [o.run(us[b], 0.01, 40)[1] for b in range(1, 6)]
    tol = 0.5 * min(h.min() for h in hist)
    s = pcf.Solver(*grid, batch=6)
    u = torch.from_numpy(us).cuda()
    before = u[0].clone()
    steps, J, jumps = s.run(u, 0.01, 36, tol=tol, dmd_period=9, dmd_snapshots=3)
    assert jumps >= 1 and steps[0] == 0
    assert torch.equal(u[0], before)
