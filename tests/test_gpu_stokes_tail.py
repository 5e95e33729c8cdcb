"""The Stokes solve of a given right-hand side keeps the tail of a decaying Chebyshev spectrum to FP64's
relative precision, coefficient by coefficient, against elimination in extended precision.

Spectrum exp(-n/2): the last coefficients are 1e-10 of the first.  Tolerance 1e-12 of the local
envelope (largest of three neighbours of one parity): 25 terms of 2^-53 each and the derivative's
weights 2 n stay below 1e-13 of it."""
import numpy as np
import pytest

import pcf_inputs as gi
from oracle import PCFOracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L = np.longdouble


def _eliminate(A, b):
    s = 1 / np.abs(A).max(1)
    A, b, n = A * s[:, None], b * s[:, None], len(A)
    for k in range(n):
        p = k + int(np.argmax(np.abs(A[k:, k])))
        A[[k, p]], b[[k, p]] = A[[p, k]], b[[p, k]]
        f = A[k + 1:, k] / A[k, k]
        A[k + 1:, k:] -= np.outer(f, A[k, k:])
        b[k + 1:] -= np.outer(f, b[k])
    x = np.zeros_like(b)
    for k in range(n - 1, -1, -1):
        x[k] = (b[k] - A[k, k + 1:] @ x[k + 1:]) / A[k, k]
    return x


def _reference(N, kx, kz, nu, step, F):
    """One mode: (1/step - nu Lap) x + grad p = F, div x = 0, x(+-1) = 0 in the unknowns (i u, v, i w, p)."""
    n1 = N + 1
    D = np.zeros((n1, n1), L)
    for n in range(1, n1):
        D[np.arange(n - 1, -1, -2), n] = 2 * n
    D[0] /= 2
    I, alt, kx, kz = np.eye(n1, dtype=L), (-1.0) ** np.arange(n1), L(kx), L(kz)
    H = (1 / (L(nu) * L(step)) + kx * kx + kz * kz) * I - D @ D
    A = np.zeros((4 * n1, 4 * n1), L)
    b = np.zeros((4 * n1, 2), L)
    G = np.stack([1j * F[0], F[1], 1j * F[2]])
    for k, (d, g) in enumerate(zip((kx * I, D, kz * I), (-kx * I, D, -kz * I))):
        r, c = slice(k * (N - 1), (k + 1) * (N - 1)), slice(k * n1, (k + 1) * n1)
        A[r, c], A[r, 3 * n1:] = H[:N - 1], g[:N - 1]
        A[3 * (N - 1) + 2 * k, c], A[3 * (N - 1) + 2 * k + 1, c] = 1, alt
        A[3 * n1:, c] = d
        b[r, 0], b[r, 1] = G[k].real[:N - 1] / L(nu), G[k].imag[:N - 1] / L(nu)
    x = _eliminate(A, b)[:3 * n1].reshape(3, n1, 2)
    x = x[..., 0] + 1j * x[..., 1]
    return np.stack([-1j * x[0], x[1], -1j * x[2]])


@pytest.mark.parametrize("batch,kind", [(1, 0), (3, 2), (9, 3)])
def test_tail_of_a_decaying_spectrum(batch, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as pcf
    pcf.load_library()
    grid, N = (16, 49, 16), 48
    o = PCFOracle(*grid, Re=1000.0, dtau_hat=0.5)
    rng = np.random.default_rng(7)
    shape = (batch,) + gi.random_perturbation(*grid, 0.1, 1).shape
    F = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * np.exp(-0.5 * np.arange(N + 1))
    F[..., N - 1:] = 0
    s = pcf.Solver(*grid, batch=batch, Re=1000.0, dtau_hat=0.5, solve_kind=kind)
    Fd = torch.from_numpy(F).cuda()
    for step, modes in ((0.25, [(1, 1), (0, 2)]), (0.5, [(7, 0)])):
        x = s.influence_matrix_solve(Fd, step).cpu().numpy()
        for i, p in modes:
            ref = _reference(N, o.kx[i], o.kz[p], 1e-3, step, F[batch - 1, :, i, p])
            a = np.abs(ref)
            env = np.maximum(a, np.maximum(np.pad(a, ((0, 0), (2, 0)))[:, :-2], np.pad(a, ((0, 0), (0, 2)))[:, 2:]))
            assert np.max(np.abs(x[batch - 1, :, i, p] - ref) / env) <= 1e-12
