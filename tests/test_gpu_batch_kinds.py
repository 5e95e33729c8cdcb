"""Batches whose problems ask for different Stokes solves (solve_kind): a problem of kind 1 has no dense
operators, so the whole batch takes the per-mode kernel.  Against the oracle at the plain FP64 bar of
1e-11, as the other batch tests."""
import ctypes

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


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("kinds", [(0, 1), (1, 0), (2, 1), (3, 1, 0), (4, 1), (5, 1), (5, 0), (0, 5)])
def test_problems_with_different_solves(pcf, kinds, precision):
    grid, lib = (16, 17, 16), pcf.load_library()
    arr = (pcf._Params * len(kinds))(*[pcf._Params(*grid, 1, pcf.LX_PAPER, pcf.LZ_PAPER, 400.0, 0.25, 0.25, precision, 0,
                                                   k, 0, 0, 0, 0, 0.0) for k in kinds])
    h = ctypes.c_void_p()
    pcf._check(lib.pcf_batch_create(arr, len(kinds), pcf._stream(), ctypes.byref(h)))
    us = gi.batch(gi.random_perturbation, range(len(kinds)), *grid, 0.1)
    u = torch.from_numpy(us).cuda()
    r, f, w = (torch.empty_like(u) for _ in range(3))
    J = torch.empty(len(kinds), dtype=torch.float64, device="cuda")
    H = torch.empty((2, len(kinds)), dtype=torch.float64, device="cuda")
    p = pcf._ptr
    pcf._check(lib.pcf_residual(h, p(u), p(r), p(J)))
    pcf._check(lib.pcf_adjoint_gradient(h, p(u), p(r), p(f)))
    pcf._check(lib.pcf_influence_matrix_solve(h, p(u), p(w), 0.25))
    pcf._check(lib.pcf_descent_step(h, p(u), 0.01, 2, p(H)))
    torch.cuda.synchronize()
    o = PCFOracle(*grid)
    for b in range(len(kinds)):
        r_ref, J_ref = o.residual(us[b])
        ref, href = o.run(us[b], 0.01, 2)
        assert _rel(r[b].cpu().numpy(), r_ref) <= TOL and abs(float(J[b]) - J_ref) <= TOL * J_ref
        assert _rel(f[b].cpu().numpy(), o.adjoint_direction(us[b], r_ref)) <= TOL
        assert _rel(w[b].cpu().numpy(), o.stokes_step(us[b], 0.25)) <= TOL
        assert _rel(u[b].cpu().numpy(), ref) <= TOL and np.max(np.abs(H[:, b].cpu().numpy() - href) / href) <= TOL
    lib.pcf_destroy(h)
