"""The FP64 forms' fixed-point per-mode kernels (k_yana_fx, k_ysolve_fx, k_ysynth_fx, k_ystep_fx)
against the oracle at the ends of their ranges: the smallest and the largest accepted ny, both
residues of N mod 4 (the unpaired row sits in the even or in the odd class), mode counts that
leave a partial tile, and group sizes 1 to 8 with a partial last group.

Tolerance: the plain FP64 bar of 1e-11.  A product's unit is 2^-55 of (largest row entry) x
(largest column value); 65 terms and the derivative's suffix sums stay below 1e-14 of the
field's largest value, and the Stokes operators' condition numbers (~1e4) are those of the
oracle's own solve."""
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


@pytest.mark.parametrize("grid,batch,group", [((16, 9, 16), 9, 8), ((16, 11, 32), 3, 2), ((16, 125, 16), 1, 0),
                                              ((16, 123, 16), 2, 0), ((32, 31, 16), 5, 4), ((48, 33, 16), 2, 1)])
def test_entry_points_and_step(pcf, grid, batch, group):
    o = PCFOracle(*grid, dtau_hat=0.5)
    us = gi.batch(gi.random_perturbation, range(80, 80 + batch), *grid, 0.1)
    u = torch.from_numpy(us).cuda()
    outs = []
    for kind in (2, 3):  # the fused half-step, and the separate kernels
        s = pcf.Solver(*grid, batch=batch, dtau_hat=0.5, modes_per_block=group, solve_kind=kind)
        r, J = s.residual(u)
        f = s.adjoint_gradient(u, r)
        w = [s.influence_matrix_solve(u, step) for step in (0.25, 0.5)]
        v = u.clone()
        H = s.descent_step(v, 0.01, 2)
        outs.append([t.cpu().numpy() for t in (r, J, f, *w, v, H)])
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*outs))
    r, J, f, w1, w2, v, H = outs[0]
    for b in {0, batch - 1}:
        r_ref, J_ref = o.residual(us[b])
        assert _rel(r[b], r_ref) <= TOL and abs(J[b] - J_ref) <= TOL * J_ref
        assert _rel(f[b], o.adjoint_direction(us[b], r_ref)) <= TOL
        assert _rel(w1[b], o.stokes_step(us[b], 0.25)) <= TOL
        assert _rel(w2[b], o.stokes_step(us[b], 0.5)) <= TOL
        ref, href = o.run(us[b], 0.01, 2)
        assert _rel(v[b], ref) <= TOL and np.max(np.abs(H[:, b] - href) / href) <= TOL


def test_a_mode_that_is_not_finite_stays_in_its_instance(pcf):
    """A NaN in the real part of one coefficient of f_v makes the real part of that mode's v NaN
    and leaves the group's other instances and the other modes alone."""
    grid = (16, 17, 16)
    us = gi.batch(gi.random_perturbation, range(90, 93), *grid, 0.1)
    s = pcf.Solver(*grid, batch=3, modes_per_block=4)
    clean = s.influence_matrix_solve(torch.from_numpy(us).cuda(), 0.25).cpu().numpy()
    us[1, 1, 2, 1, 5] = np.nan
    got = s.influence_matrix_solve(torch.from_numpy(us).cuda(), 0.25).cpu().numpy()
    assert np.isnan(got[1, 1, 2, 1].real).all()
    got[1, :, 2, 1] = clean[1, :, 2, 1]
    assert np.array_equal(got, clean)


@pytest.mark.parametrize("grids", [[(64, 9, 64, 1)], [(64, 13, 64, 4)], [(64, 21, 64, 1), (16, 13, 16, 2)],
                                   [(128, 9, 64, 1), (96, 11, 96, 1), (16, 9, 16, 1)]])
def test_launch_shapes_give_the_same_bits(pcf, grids):
    """The thread counts, tiles and groups a batch chooses move no bit: every sum is an exact
    integer sum.  Many small CTAs (96 and 128 threads), tiles of 16 modes, planes of unequal
    sizes in one launch, each against its instances one by one."""
    us = [gi.random_perturbation(*g[:3], 0.1, 60 + k) for g in grids for k in range(g[3])]
    s = pcf.Solver.batched(grids, solve_kind=3)
    u = torch.from_numpy(np.concatenate([x.ravel() for x in us])).cuda()
    H = s.descent_step(u, 0.01, 1).cpu().numpy()
    got = u.cpu().numpy()
    for b, x in enumerate(us):
        one = pcf.Solver(*s.grids[b][:3], batch=1, solve_kind=3)
        v = torch.from_numpy(x[None]).cuda()
        h = one.descent_step(v, 0.01, 1).cpu().numpy()
        assert np.array_equal(got[s.offsets[b]:s.offsets[b + 1]], v.cpu().numpy().ravel())
        assert np.array_equal(H[:, b], h[:, 0])
        one.close()
    s.close()
