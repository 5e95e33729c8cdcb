"""DMD extrapolation where its parts change over: snapshot counts around the row blocks of the
tall-skinny QR (k_tsqr) and beyond the columns it serves, contexts of one and of several
instances (the candidates' residuals run in a batch of their own), and grids of both parities.

Affine dynamics with five decaying directions, as in the other DMD tests: the snapshot matrix
has rank six, the steady state agrees with the oracle's SVD-based DMD to 1e-9."""
import numpy as np
import pytest

import pcf_inputs as gi
from oracle import PCFOracle, dmd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


@pytest.fixture(scope="module")
def pcf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("grid,M,batch", [((16, 9, 16), 7, 1), ((16, 11, 16), 30, 3), ((32, 17, 16), 63, 1),
                                          ((16, 17, 16), 64, 2), ((16, 11, 16), 124, 1)])
def test_dmd_snapshot_counts(pcf, grid, M, batch):
    o = PCFOracle(*grid)
    rng = np.random.default_rng(M)
    star = o.to_psi(gi.random_perturbation(*grid, 0.05, M))
    Q, _ = np.linalg.qr(rng.standard_normal((o.psi_dim(), 5)))
    a, mu = 0.01 * rng.standard_normal(5), np.linspace(0.5, 0.95, 5)
    S = np.stack([star + Q @ (a * mu ** k) for k in range(M + 1)])
    s = pcf.Solver(*grid, batch=batch)
    Sd = torch.from_numpy(S).cuda()
    out, r, J = s.dmd_extrapolate(Sd, rank_tol=1e-10)
    psi, r_ref, costs = dmd.dmd_extrapolate(S.T, lambda p: o.residual(o.from_psi(p))[1], rank_tol=1e-10)
    assert r == r_ref and abs(J - costs[r_ref]) <= 1e-9 * costs[r_ref]
    assert _rel(out.cpu().numpy(), o.from_psi(psi)) <= 1e-9
    again, r2, J2 = s.dmd_extrapolate(Sd, rank_tol=1e-10)
    assert r2 == r and J2 == J and torch.equal(out, again)
