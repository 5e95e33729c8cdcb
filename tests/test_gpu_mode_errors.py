"""Rounding of the FP64 forms mode by mode on a large plane with a flat spectrum, against the residual
in extended precision (numpy's longdouble): every Fourier mode of r1 keeps the relative precision that
FP64 transforms would give it, not only the field's norm.

Tolerance: a mode of r1 is the difference of two values near 1/dt = 4 of the state and six products of
two transforms each, of 14 levels of 2^-54 rounding each: 4 x 2^-54 + sqrt(6 x 3 x 14) x 2^-54, about 20
x 2^-54 = 1.1e-15; 1.5e-15 for the median of the modes."""
import numpy as np
import pytest

from oracle import PCFOracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, C = np.longdouble, np.clongdouble


def _residual(o, u, step=0.25):
    """r1 = (u^step - u)/step of plane Couette flow, with the oracle's layout and wavenumbers."""
    N, n1, nx, nz = o.N, o.N + 1, o.nx, o.nz
    n = np.arange(n1)
    T = np.cos(L("3.14159265358979323846264338327950288") * (np.outer(n, n) % (2 * N)).astype(L) / N)
    c = np.where((n == 0) | (n == N), L(2), L(1))
    Ti = L(2) / (N * np.outer(c, c)) * T.T
    D, y = o.Dmat.astype(L), T[:, 1][:, None, None]
    kx, kz, nu, u = o.kx.astype(L)[:, None, None], o.kz.astype(L)[None, :, None], 1 / L(400), u.astype(C)

    def cheb(a, M):
        return (a.real @ M.T) + 1j * (a.imag @ M.T)

    def phys(a):
        v = np.moveaxis(cheb(a, T), -1, -3)
        full = np.zeros(v.shape[:-2] + (nx, nz // 2 + 1), C)
        full[..., o.x_index, :o.Mz] = v
        return np.fft.irfft2(full, s=(nx, nz), norm="forward")
    v = phys(u)
    F = np.empty_like(u)
    for i in range(3):
        m = -(y + v[0]) * phys(1j * kx * u[i]) - v[1] * phys(cheb(u[i], D)) - v[2] * phys(1j * kz * u[i])
        if i == 0:
            m -= v[1]
        F[i] = cheb(np.moveaxis(np.fft.rfft2(m, norm="forward")[..., o.x_index, :o.Mz], -3, -1), Ti)
    F = (F + u / L(step)) / nu
    # one system per mode in (i u, v, i w, p)
    k1, k3 = (a.reshape(-1, 1, 1)[1:] for a in np.broadcast_arrays(kx[..., 0], kz[..., 0]))
    I, alt, D2 = np.eye(n1, dtype=L), (-1.0) ** n, D @ D
    H = (1 / (nu * L(step)) + k1 * k1 + k3 * k3) * I - D2
    A = np.zeros((len(k1), 4 * n1, 4 * n1), L)
    for k, (d, g) in enumerate(((k1 * I, -k1 * I), (D + 0 * H, D + 0 * H), (k3 * I, -k3 * I))):
        r, q = slice(k * (N - 1), (k + 1) * (N - 1)), slice(k * n1, (k + 1) * n1)
        A[:, r, q], A[:, r, 3 * n1:] = H[:, :N - 1], g[:, :N - 1]
        A[:, 3 * (N - 1) + 2 * k, q], A[:, 3 * (N - 1) + 2 * k + 1, q] = 1, alt
        A[:, 3 * n1:, q] = d
    G = np.stack([1j * F[0], F[1], 1j * F[2]]).reshape(3, -1, n1)[:, 1:, :N - 1]
    b = np.zeros((len(k1), 4 * n1, 2), L)
    b[:, :3 * (N - 1), 0] = np.concatenate(list(G.real), -1)
    b[:, :3 * (N - 1), 1] = np.concatenate(list(G.imag), -1)
    s = 1 / np.abs(A).max(-1, keepdims=True)
    A, b, x = A * s, b * s, np.zeros_like(b)
    A64 = np.linalg.inv(A.astype(float))
    for _ in range(4):
        x = x + A64 @ (b - A @ x).astype(float)
    x = (x[..., 0] + 1j * x[..., 1])[:, :3 * n1].reshape(-1, 3, n1)
    out = np.zeros((3, o.Mx * o.Mz, n1), C)
    out[0, 1:], out[1, 1:], out[2, 1:] = -1j * x[:, 0], x[:, 1], -1j * x[:, 2]
    return ((out.reshape(u.shape) - u) / L(step)).astype(complex)


def test_modes_of_a_flat_spectrum():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as pcf
    pcf.load_library()
    grid = (128, 9, 128)
    o = PCFOracle(*grid)
    u = o.from_psi(1e-3 * np.random.default_rng(6).standard_normal(o.psi_dim()))
    s = pcf.Solver(*grid)
    r = s.residual(torch.from_numpy(u[None]).cuda())[0].cpu().numpy()[0]
    ref = _residual(o, u)
    e = np.sqrt((np.abs(r - ref) ** 2).sum((0, 3)) / (np.abs(ref) ** 2).sum((0, 3))).ravel()[1:]
    assert np.median(e) <= 1.5e-15
