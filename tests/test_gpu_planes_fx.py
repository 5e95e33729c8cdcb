"""The FP64 forms' fixed-point plane transforms (k_synth_fx, k_prod_fx) against the oracle at
every transform length in x and in z, and at the ends of the FP64 range.

Tolerance: the residual and the descent direction are linear images of transforms whose unit
is 2^-60 of the sum of the magnitudes that enter them, below FP64's rounding; the plain FP64
bar of 1e-11 (Stokes operators with condition numbers up to ~1e4) applies unchanged."""
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


@pytest.mark.parametrize("grid", [(16, 9, 128), (128, 9, 16), (48, 11, 96), (96, 9, 48), (64, 15, 32), (32, 9, 64),
                                  (128, 9, 128), (96, 11, 96)])
def test_every_transform_length(pcf, grid):
    o = PCFOracle(*grid)
    u0 = gi.random_perturbation(*grid, 0.1, 71)
    s = pcf.Solver(*grid, batch=1)
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


@pytest.mark.parametrize("scale", [2.0 ** -400, 2.0 ** -60, 2.0 ** 60, 2.0 ** 200])
def test_states_of_any_size(pcf, scale):
    """Block exponents follow the data: tiny states (the terms linear in u remain) and huge ones
    (the quadratic terms dominate)."""
    grid = (32, 17, 16)
    o = PCFOracle(*grid)
    u0 = scale * gi.random_perturbation(*grid, 0.1, 72)
    s = pcf.Solver(*grid, batch=1)
    r, _ = s.residual(torch.from_numpy(u0[None]).cuda())
    r_ref, _ = o.residual(u0)
    assert _rel(r.cpu().numpy()[0] / scale, r_ref / scale) <= TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_value_that_is_not_finite_reaches_the_norm(pcf, bad):
    """One such coefficient in one instance makes that instance's J not finite and leaves its
    neighbour alone."""
    grid = (16, 17, 16)
    u0 = gi.batch(gi.random_perturbation, [73, 74], *grid, 0.1)
    o = PCFOracle(*grid)
    clean = u0[1].copy()
    u0[0, 0, 1, 2, 3] = bad
    s = pcf.Solver(*grid, batch=2)
    r, J = s.residual(torch.from_numpy(u0).cuda())
    assert not np.isfinite(float(J[0]))
    r_ref, J_ref = o.residual(clean)
    assert abs(float(J[1]) - J_ref) <= TOL * J_ref
    assert _rel(r.cpu().numpy()[1], r_ref) <= TOL


@pytest.mark.parametrize("low,high", [(-300, 300), (-70, 0), (0, 150), (-990, -900)])
def test_bound_of_a_plane_with_a_wide_range(pcf, low, high):
    """The block exponent comes from a running single-precision sum with a moving reference:
    modes spread over hundreds of binary orders, in any order, and a mean far above or below the
    modes that enter a derivative."""
    grid = (32, 9, 16)
    rng = np.random.default_rng(5)
    u0 = gi.random_perturbation(*grid, 0.1, 74)
    o = PCFOracle(*grid)
    s = pcf.Solver(*grid, batch=1)
    e = rng.integers(low, high, size=u0.shape[1:3])
    for i in range(1, (e.shape[0] + 1) // 2):
        e[-i, 0] = e[i, 0]  # the modes p = 0 stay Hermitian in m
    for mean in (low, high):
        e[0, 0] = mean
        v = u0 * 2.0 ** (e[None, :, :, None] - max(0.0, high))
        r, _ = s.residual(torch.from_numpy(v[None]).cuda())
        assert _rel(r.cpu().numpy()[0], o.residual(v)[0]) <= TOL
        if low >= -300:  # the norm's square stays in range
            assert abs(float(s.norm(torch.from_numpy(v[None]).cuda())[0]) - o.norm(v)) <= TOL * o.norm(v)
