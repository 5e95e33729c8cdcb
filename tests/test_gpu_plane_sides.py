"""The FP64 forms on planes with a side of 18, 24, 36, 54, 72 or 108 (transform lengths that are not
8 times 2, 4, 6, 8, 12 or 16), alone, next to the other lengths and in one batch with them, against
the oracle.

Tolerance: the plain FP64 bar of 1e-11 of the other plane tests."""
import numpy as np
import pytest

import pcf_inputs as gi
from oracle import PCFOracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-11


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


@pytest.fixture(scope="module")
def pcf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("grid,precision", [((24, 33, 24), 0), ((24, 33, 24), 2), ((72, 9, 36), 0), ((18, 9, 54), 0),
                                            ((18, 9, 54), 2), ((108, 9, 18), 0), ((36, 11, 72), 0), ((54, 9, 108), 0),
                                            ((24, 9, 128), 0), ((128, 9, 24), 0), ((18, 9, 16), 0), ((32, 9, 36), 0),
                                            ((108, 9, 108), 0)])
def test_residual_gradient_norm(pcf, grid, precision):
    o = PCFOracle(*grid)
    u0 = gi.random_perturbation(*grid, 0.1, 75)
    s = pcf.Solver(*grid, batch=1, precision=precision)
    u = torch.from_numpy(u0[None]).cuda()
    r, J = s.residual(u)
    f = s.adjoint_gradient(u, r)
    r_ref, J_ref = o.residual(u0)
    f_ref = o.adjoint_direction(u0, r_ref)
    for c in range(3):
        assert _rel(r.cpu().numpy()[0, c], r_ref[c]) <= TOL
        assert _rel(f.cpu().numpy()[0, c], f_ref[c]) <= TOL
    assert abs(float(J[0]) - J_ref) <= TOL * J_ref
    assert abs(float(s.norm(u)[0]) - o.norm(u0)) <= TOL * o.norm(u0)


def test_batch_of_sides(pcf):
    """One launch over planes of every kind of side: each instance as the oracle has it."""
    grids = [(24, 9, 18, 2), (32, 9, 16, 1), (128, 9, 64, 1), (72, 9, 54, 1)]
    us = [gi.random_perturbation(*g[:3], 0.1, 40 + k) for g in grids for k in range(g[3])]
    s = pcf.Solver.batched(grids)
    u = torch.from_numpy(np.concatenate([x.ravel() for x in us])).cuda()
    H = s.descent_step(u, 0.001, 3).cpu().numpy()
    for b, x in enumerate(us):
        ref, href = PCFOracle(*s.grids[b][:3]).run(x, 0.001, 3)
        assert _rel(s.view(u, b).cpu().numpy(), ref) <= TOL and np.max(np.abs(H[:, b] - href) / href) <= TOL


def test_dns(pcf):
    grid = (36, 9, 24)
    o = PCFOracle(*grid, dt=0.005, dtau_hat=0.005)
    u0 = gi.random_perturbation(*grid, 0.1, 41)
    s = pcf.Solver(*grid, batch=1, dt=0.005, dtau_hat=0.005)
    u = torch.from_numpy(u0[None]).cuda()
    H, _, _ = s.dns(u, 4, max_guesses=0)
    v, norms = u0.copy(), []
    for _ in range(4):
        norms.append(o.norm(v))
        v = v + o.dt * o.residual(v)[0]
    assert _rel(u.cpu().numpy()[0], v) <= TOL
    assert np.max(np.abs(H.cpu().numpy()[:, 0] - norms) / np.array(norms)) <= TOL
