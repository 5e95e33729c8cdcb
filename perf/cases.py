"""Workloads of the adjoint-descent framework, through its public entry points.

A case names one call (or the pair of calls a user makes together), its grid, batch and
options.  The grids are Fourier(x) x Chebyshev(y) x Fourier(z) with 2/3 dealiasing; states are
complex128 [batch][3][Mx][Mz][ny] coefficients of perturbations of the laminar flow.

kinds:
  step       Solver.descent_step on a device state, in place
  step_host  Solver.descent_step_host: the same with a pinned host state
  gradient   Solver.residual, then Solver.adjoint_gradient
  stokes     Solver.influence_matrix_solve
  dns        Solver.dns: the Stokes step as a time stepper, with guesses at extrema of ||u||
  uneven     Solver.batched(...).descent_step over instances of several grids
  dmd        Solver.dmd_extrapolate on stored snapshots
  fno        FNO.loss_grad: loss and parameter gradient of the learned proposal
"""
import math

import numpy as np
import torch

import paper_2306_00165_gb300 as pcf

SIZES = (16, 32, 48, 64, 96, 128)      # accepted nx, nz
COUETTE, POISEUILLE, ASBL = 0, 1, 2
FP64, MIXED, FLOAT_FLOAT = 0, 1, 2
UNEVEN = ((32, 33, 32), (48, 49, 48), (64, 65, 64))


def _case(kind, nx, ny, nz, batch, **kw):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "batch": batch, "Re": 400.0, "precision": FP64,
         "base_flow": COUETTE, "symmetry": 0, "nsteps": 1, "dtau": 0.01}
    c.update(kw)
    return c


def listed():
    return [
        # one guess on the smallest grid, state on the host: latency, launches and copies
        dict(_case("step_host", 16, 17, 16, 1), name="step_host_16"),
        # the benchmark's step: eight streak/roll guesses advanced together
        dict(_case("step", 32, 33, 32, 8), name="step_32x8"),
        # the float-float form of the same workload, a few steps per call
        dict(_case("step", 32, 33, 32, 8, precision=FLOAT_FLOAT, nsteps=4), name="step_ff_32x8"),
        # descent kept in the s1,s2-symmetric subspace
        dict(_case("step", 32, 33, 32, 8, symmetry=3, nsteps=4), name="step_sym_32x8"),
        # residual and descent direction of plane Poiseuille flow at the middle resolution
        dict(_case("gradient", 64, 65, 64, 2, base_flow=POISEUILLE), name="gradient_64x2"),
        # residual and descent direction of one guess on the largest grid, FP64
        dict(_case("gradient", 128, 97, 128, 1, Re=1000.0), name="gradient_128"),
        # the mixed form's workload: FP32 planes, split-BF16 Chebyshev transforms
        dict(_case("step", 128, 97, 128, 1, Re=1000.0, precision=MIXED, dtau=0.001, nsteps=2), name="step_mixed_128"),
        # 64 guesses of uneven grids in one context (24 + 24 + 16)
        dict(_case("uneven", 0, 0, 0, 64, n32=24, n48=24, n64=16), name="step_uneven_64"),
        # the Stokes solve alone on a ragged grid (ny - 1 = 30 is 2 mod 4)
        dict(_case("stokes", 96, 31, 48, 3), name="stokes_96x31x48"),
        # DNS that makes the guesses of the robustness experiment
        dict(_case("dns", 32, 33, 32, 4, nsteps=64), name="dns_32x4"),
        # DMD jump of one instance from 20 stored snapshots
        dict(_case("dmd", 32, 33, 32, 1, snapshots=20), name="dmd_32"),
        # one training gradient of the learned proposal: 190 modes, 32 samples
        dict(_case("fno", 32, 33, 32, 32), name="fno_grad_32"),
    ]


def _points(c):
    return c["nx"] * c["ny"] * c["nz"] * c["batch"]


def _odd(rng, lo, hi):
    """An odd ny in lo..hi, spread over its logarithm."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, v | 1))


def _grid(rng, most, ny_hi=97):
    """A grid whose points are at most `most`, small ones as likely as large ones."""
    cap = math.exp(rng.uniform(math.log(4096), math.log(most)))
    while True:
        nx, nz, ny = rng.choice(SIZES), rng.choice(SIZES), _odd(rng, 9, ny_hi)
        if cap / 6 <= nx * ny * nz <= cap or (nx == nz == 16 and nx * ny * nz <= 2 * cap):
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(["step", "step", "step", "gradient", "gradient", "gradient", "step_host", "stokes", "dns",
                       "uneven", "dmd", "fno"])
    if kind == "uneven":
        return _case("uneven", 0, 0, 0, 0, n32=rng.randint(1, 24), n48=rng.randint(0, 24), n64=rng.randint(0, 16),
                     nsteps=1)
    if kind == "fno":
        nx, ny, nz = _grid(rng, 70000, 49)
        return _case("fno", nx, ny, nz, rng.choice([1, 8, 16, 32, 48]))
    if kind == "dmd":
        nx, ny, nz = _grid(rng, 120000, 65)
        return _case("dmd", nx, ny, nz, 1, snapshots=rng.randint(5, 24))
    nx, ny, nz = _grid(rng, 1600000)
    c = _case(kind, nx, ny, nz, 1)
    most = 1600000 if kind in ("step", "gradient", "step_host") else 1000000
    room = max(1, most // (nx * ny * nz))
    c["batch"] = min(room, 16, max(1, int(round(math.exp(rng.uniform(0.0, math.log(16.5)))))))
    if kind in ("step", "dns"):
        left = max(1, most // _points(c))
        c["nsteps"] = min(left, 64 if kind == "dns" else 16, rng.choice([1, 2, 5, 16, 64]))
    c["base_flow"] = rng.choice([COUETTE, COUETTE, POISEUILLE, ASBL])
    if kind in ("step", "gradient") and nx * ny * nz >= 16 * 17 * 16:
        c["precision"] = rng.choice([FP64, FP64, FP64, MIXED, FLOAT_FLOAT])
    if kind == "step" and c["precision"] == FP64:
        c["symmetry"] = rng.choice([0, 0, 2, 3]) if c["base_flow"] == COUETTE else rng.choice([0, 2])
    if max(nx, nz) >= 96:                  # the explicit Euler step on fine grids
        c["Re"], c["dtau"] = 1000.0, 0.001
    return c


# ---------------------------------------------------------------- inputs
def _steps(c):
    """(dt, dtau_hat) of a case: the paper's 0.25, or the DNS step."""
    return (0.005, 0.005) if c["kind"] == "dns" else (0.25, 0.25)


def _dims(nx, nz):
    Kx, Kz = nx // 3 - 1, nz // 3 - 1
    return Kx, Kz, 2 * Kx + 1, Kz + 1


def _waves(nx, nz, dev):
    """m and p of the stored modes, kx and kz in the paper's box."""
    Kx, Kz, Mx, Mz = _dims(nx, nz)
    m = torch.tensor(list(range(Kx + 1)) + list(range(-Kx, 0)), dtype=torch.float64, device=dev)
    p = torch.arange(Mz, dtype=torch.float64, device=dev)
    return m, p, 1.14 * m, 2.5 * p


def _deriv(n1, dev):
    """Matrix of d/dy on Chebyshev coefficients."""
    D = np.zeros((n1, n1))
    for n in range(1, n1):
        for k in range(n - 1, -1, -2):
            D[k, n] = 2.0 * n if k > 0 else 1.0 * n
    return torch.from_numpy(D).to(dev)


def _times(n1, series, drop, dev):
    """Matrix of multiplication by an even series sum_j c_j T_2j, the input's top `drop` coefficients cut."""
    W = np.zeros((n1, n1))
    for i in range(n1 - drop):
        for j, cj in enumerate(series):
            W[i + 2 * j, i] += 0.5 * cj
            W[abs(i - 2 * j), i] += 0.5 * cj
    return torch.from_numpy(W).to(dev)


def _field(nx, ny, nz, batch, amplitude, seed, dev="cuda"):
    """Random divergence-free, no-slip perturbations with coefficient variance ~ exp(-|(m, p, n)|)
    and about the given volume-mean norm, as complex128 [batch][3][Mx][Mz][ny]."""
    g = torch.Generator(device=dev).manual_seed(seed)
    Kx, Kz, Mx, Mz = _dims(nx, nz)
    m, p, kx, kz = _waves(nx, nz, dev)
    n = torch.arange(ny, dtype=torch.float64, device=dev)
    sd = torch.exp(-0.5 * torch.sqrt(m[:, None, None] ** 2 + p[None, :, None] ** 2 + n ** 2))

    def noise():
        a = torch.randn((batch, Mx, Mz, ny, 2), dtype=torch.float64, device=dev, generator=g)
        return torch.view_as_complex(a) * sd

    def hermitian(a):
        a[:, Kx + 1:, 0] = a[:, 1:Kx + 1, 0].flip(1).conj()
        a[:, 0, 0] = a[:, 0, 0].real.to(a.dtype)
        return a

    W1 = _times(ny, (0.5, -0.5), 2, dev).to(torch.complex128)         # 1 - y^2
    W2 = _times(ny, (0.375, -0.5, 0.125), 4, dev).to(torch.complex128)  # (1 - y^2)^2
    v, eta = hermitian(noise() @ W2.T), hermitian(noise() @ W1.T)
    mean = (noise()[:, 0, :2].real.to(torch.complex128) if Mz > 1 else noise()[:, :2, 0]) @ W1.T
    KX, KZ = kx[:, None, None], kz[None, :, None]
    k2 = KX ** 2 + KZ ** 2
    k2[0, 0] = 1.0
    xi = -(v @ _deriv(ny, dev).to(torch.complex128).T)
    out = torch.stack([(-1j * KX * xi - 1j * KZ * eta) / k2, v, (-1j * KZ * xi + 1j * KX * eta) / k2], 1)
    out[:, :, 0, 0] = 0
    out[:, 0, 0, 0] = mean[:, 0].real.to(out.dtype)
    out[:, 2, 0, 0] = mean[:, 1].real.to(out.dtype)
    val = (out @ _nodes(ny, dev).T.to(torch.complex128)).abs().square()
    val[:, :, :, 1:] *= 2
    w = torch.from_numpy(_cc(ny - 1)).to(dev)
    norm = torch.sqrt(0.5 * (val.sum((1, 2, 3)) * w).sum(-1))
    return (out * (amplitude / norm)[:, None, None, None, None]).contiguous()


def _snapshots(c, seed, dev="cuda"):
    """Snapshot vectors near a slow state: a fixed part, five decaying parts, small noise in each."""
    g = torch.Generator(device=dev).manual_seed(seed + 77)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    parts = torch.stack([_psi(nx, ny, nz, _field(nx, ny, nz, 1, 0.1, seed + k)[0]) for k in range(6)])
    k = torch.arange(c["snapshots"], dtype=torch.float64, device=dev)
    mu = torch.linspace(0.5, 0.95, 5, dtype=torch.float64, device=dev)
    S = parts[0] + (0.2 * mu[None, :] ** k[:, None]) @ parts[1:]
    size = parts[0].abs() + parts[1].abs()
    return (S + 1e-3 * size * torch.randn(S.shape, dtype=torch.float64, device=dev, generator=g)).contiguous()


def _params(MP, ny, seed, W=32, L=4):
    """Parameters of the proposal network in the library's layout: {name: float32 array}."""
    rng = np.random.default_rng(seed)
    F = 4 * ny

    def normal(shape, s):
        return (rng.standard_normal(shape, dtype=np.float32) * np.float32(s)).astype(np.float32)
    p = {"E": normal((MP, W, F), F ** -0.5), "bE": normal((W,), 0.02), "D": normal((MP, F, W), 0.1 * W ** -0.5),
         "bD": normal((MP, F), 0.02)}
    for l in range(L):
        p[f"R{l}"], p[f"L{l}"] = normal((MP, W, W), 0.5 * W ** -0.5), normal((W, W), 0.5 * W ** -0.5)
        p[f"b{l}"] = normal((W,), 0.02)
    return p


def _pairs(c, seed, dev="cuda"):
    """Scaled features and the increments to learn, float32 [MP][S][ny][4]."""
    Kx, Kz, Mx, Mz = _dims(c["nx"], c["nz"])
    g = torch.Generator(device=dev).manual_seed(seed)
    X = torch.randn((Mx * Mz, c["batch"], c["ny"], 4), device=dev, generator=g)
    return X, 0.1 * torch.randn(X.shape, device=dev, generator=g) - 0.05 * X


def _uneven(c):
    return [(*g, c[k]) for g, k in zip(UNEVEN, ("n32", "n48", "n64")) if c[k] > 0]


def _amplitude(c):
    return 0.2 if c["kind"] == "dns" else 0.1


def prepare(case, seed):
    c = case
    if c["kind"] == "fno":
        Kx, Kz, Mx, Mz = _dims(c["nx"], c["nz"])
        net = pcf.FNO(Mx * Mz, c["ny"], seed=0)
        net.set_params(np.concatenate([a.ravel() for a in _params(Mx * Mz, c["ny"], seed).values()]))
        X, T = _pairs(c, seed)
        return {"c": c, "net": net, "X": X, "T": T}
    if c["kind"] == "uneven":
        s = pcf.Solver.batched(_uneven(c), Re=c["Re"])
        u = torch.cat([_field(*g, 0.1, seed + k).reshape(-1) for k, g in enumerate(_uneven(c))])
        return {"c": c, "s": s, "u": u}
    dt, dh = _steps(c)
    s = pcf.Solver(c["nx"], c["ny"], c["nz"], batch=c["batch"], Re=c["Re"], dt=dt, dtau_hat=dh,
                   precision=c["precision"], base_flow=c["base_flow"], symmetry=c["symmetry"],
                   suction_length=0.5 if c["base_flow"] == ASBL else 0.0)
    st = {"c": c, "s": s}
    if c["kind"] == "dmd":
        st["S"] = _snapshots(c, seed)
        return st
    u = _field(c["nx"], c["ny"], c["nz"], c["batch"], _amplitude(c), seed)
    if c["kind"] == "step_host":
        st["u"] = u.cpu().pin_memory()
        st["J"] = torch.empty((c["nsteps"], c["batch"]), dtype=torch.float64).pin_memory()
    else:
        st["u"] = u
    return st


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "fno":
        loss, grad = state["net"].loss_grad(state["X"], state["T"])
        return {"loss": loss, "grad": grad}
    s = state["s"]
    if kind == "dmd":
        u, rank, J = s.dmd_extrapolate(state["S"], rank_tol=1e-10)
        return {"u": u, "rank": rank, "J": J}
    u = state["u"]
    if kind in ("step", "uneven"):
        J = s.descent_step(u, c["dtau"], c["nsteps"])
        return {"u": u, "J": J}
    if kind == "step_host":
        s.descent_step_host(u, c["dtau"], c["nsteps"], state["J"])
        return {"u": u, "J": state["J"]}
    if kind == "gradient":
        r, J = s.residual(u)
        return {"r": r, "J": J, "f": s.adjoint_gradient(u, r)}
    if kind == "stokes":
        return {"u": s.influence_matrix_solve(u, 0.25)}
    H, G, n = s.dns(u, c["nsteps"], max_guesses=2)
    return {"u": u, "norm": H, "guesses": G, "found": n}


# ---------------------------------------------------------------- work of one pass
def _fft(L):
    return 5.0 * L * math.log2(L)


def _flops(nx, ny, nz, kind):
    """Algorithmic flops of one instance: FFTs 5 L log2 L, folded Chebyshev matrices, tau sweeps."""
    Kx, Kz, Mx, Mz = _dims(nx, nz)
    nm, H = Mx * Mz, (ny - 1) // 2 + 1
    plane = Mz * _fft(nx) + (nx // 2) * _fft(nz)
    cheb = 4.0 * H * (2 * H - 1)
    solve = nm * (120.0 * H + 24.0 * ny)
    if kind == "stokes":
        return solve
    primal = ny * (14 * plane + 3 * nx * nz * 8.0) + nm * 8 * cheb + solve
    if kind == "dns":
        return primal
    return primal + ny * (14 * plane + 3 * nx * nz * 14.0) + nm * 8 * cheb + solve


def work(case):
    c = case
    if c["kind"] == "uneven":
        n = b = 0
        for nx, ny, nz, k in _uneven(c):
            Kx, Kz, Mx, Mz = _dims(nx, nz)
            n += k * _flops(nx, ny, nz, "step")
            b += k * 2 * 3 * Mx * Mz * ny * 16
        return {"bytes": b, "flops": n * c["nsteps"]}
    Kx, Kz, Mx, Mz = _dims(c["nx"], c["nz"])
    nm, ny = Mx * Mz, c["ny"]
    state = c["batch"] * 3 * nm * ny * 16
    if c["kind"] == "fno":
        F, W, L, S = 4 * ny, 32, 4, c["batch"]
        weights = nm * (2 * W * F + F + L * W * W) + W + L * (W * W + W)
        return {"bytes": 8 * weights + 8 * nm * S * F, "flops": nm * S * (10.0 * W * F + L * 6.0 * W * W)}
    if c["kind"] == "dmd":
        psi = nm // 2 * 2 * (4 * ny - 12)
        M = c["snapshots"]
        return {"bytes": 8 * M * psi + state, "flops": 2.0 * psi * M * M + M * _flops(c["nx"], ny, c["nz"], "dns")}
    f = c["batch"] * c["nsteps"] * _flops(c["nx"], ny, c["nz"], c["kind"])
    out = {"gradient": 3}.get(c["kind"], 2)
    return {"bytes": out * state, "flops": f}


# ---------------------------------------------------------------- the same in plain torch, 64 bits
def _nodes(ny, dev):
    n = np.arange(ny)
    return torch.from_numpy(np.cos(math.pi * (np.outer(n, n) % (2 * (ny - 1))) / (ny - 1))).to(dev)


def _cc(N):
    """Clenshaw-Curtis weights on the Gauss-Lobatto points."""
    th = math.pi * np.arange(N + 1) / N
    w = np.ones(N + 1)
    for k in range(1, N // 2 + 1):
        w -= (1.0 if 2 * k == N else 2.0) / (4.0 * k * k - 1.0) * np.cos(2.0 * k * th)
    w *= 2.0 / N
    w[0] *= 0.5
    w[N] *= 0.5
    return w


class _Plain:
    """The method's steps in plain torch: cuFFT, dense Chebyshev matrices, one LU per mode."""

    def __init__(self, nx, ny, nz, Re, dt, dh, base_flow=COUETTE, delta=0.5, dev="cuda"):
        self.nx, self.ny, self.nz, self.nu, self.dt, self.dh, self.dev = nx, ny, nz, 1.0 / Re, dt, dh, dev
        self.Kx, self.Kz, self.Mx, self.Mz = _dims(nx, nz)
        self.m, self.p, self.kx, self.kz = _waves(nx, nz, dev)
        self.bins = (self.m.long() % nx)
        self.C = _nodes(ny, dev)
        self.Ci = torch.linalg.inv(self.C)
        self.D = _deriv(ny, dev)
        self.w = torch.from_numpy(_cc(ny - 1)).to(dev)
        y = torch.cos(math.pi * torch.arange(ny, dtype=torch.float64, device=dev) / (ny - 1))
        e = torch.exp(-(1.0 + y) / delta)
        U, dU, self.V = {COUETTE: (y, torch.ones_like(y), 0.0), POISEUILLE: (1 - y * y, -2 * y, 0.0),
                         ASBL: (1 - e, e / delta, -self.nu / delta)}[base_flow]
        self.U, self.dU = U[:, None, None], dU[:, None, None]
        self.lu = {}

    def mul(self, a, A):
        """A applied to the Chebyshev index of a complex array."""
        return torch.view_as_complex(torch.stack([a.real @ A.T, a.imag @ A.T], -1))

    def phys(self, a):
        v = self.mul(a, self.C).movedim(-1, -3)
        full = torch.zeros(v.shape[:-2] + (self.nx, self.nz // 2 + 1), dtype=torch.complex128, device=self.dev)
        full[..., self.bins, : self.Mz] = v
        return torch.fft.irfft2(full, s=(self.nx, self.nz), norm="forward")

    def spec(self, f):
        F = torch.fft.rfft2(f, norm="forward")[..., self.bins, : self.Mz]
        return self.mul(F.movedim(-3, -1), self.Ci)

    def grad(self, a):
        """d_j of one component: x, y, z."""
        return [self.phys(1j * self.kx[:, None, None] * a), self.phys(self.mul(a, self.D)),
                self.phys(1j * self.kz[None, :, None] * a)]

    def factor(self, sigma):
        """LU of every mode's tau system in the real unknowns (i u, v, i w, P)."""
        if sigma in self.lu:
            return self.lu[sigma]
        n1, N, dev = self.ny, self.ny - 1, self.dev
        I, D = torch.eye(n1, dtype=torch.float64, device=dev), self.D
        D2, alt = D @ D, (-1.0) ** torch.arange(n1, dtype=torch.float64, device=dev)
        KX, KZ = torch.meshgrid(self.kx, self.kz, indexing="ij")
        KX, KZ = KX.reshape(-1)[1:], KZ.reshape(-1)[1:]      # every mode but the mean
        B = KX.numel()
        A = torch.zeros((B, 4 * n1, 4 * n1), dtype=torch.float64, device=dev)
        H = (sigma + KX ** 2 + KZ ** 2)[:, None, None] * I - D2
        div = [KX[:, None, None] * I, D.expand(B, n1, n1), KZ[:, None, None] * I]
        gr = [-div[0], div[1], -div[2]]
        for k in range(3):
            r, c = slice(k * (N - 1), (k + 1) * (N - 1)), slice(k * n1, (k + 1) * n1)
            A[:, r, c], A[:, r, 3 * n1:] = H[:, : N - 1], gr[k][:, : N - 1]
            A[:, 3 * (N - 1) + 2 * k, c], A[:, 3 * (N - 1) + 2 * k + 1, c] = 1.0, alt
            A[:, 3 * n1:, c] = div[k]
        scale = 1.0 / A.abs().amax(-1)
        A *= scale[:, :, None]
        M = sigma * I - D2
        M[N - 1], M[N] = 1.0, alt
        self.lu[sigma] = (A, scale, torch.linalg.lu_factor(A), M)
        return self.lu[sigma]

    def stokes(self, F, step):
        """(1/step - nu Lap) out + grad p = F, div out = 0, out(+-1) = 0; F [B][3][Mx][Mz][ny]."""
        A, scale, lu, M = self.factor(1.0 / (self.nu * step))
        n1, N, nb = self.ny, self.ny - 1, F.shape[0]
        F = F / self.nu
        G = F.reshape(nb, 3, -1, n1)[:, :, 1:].clone()
        G[:, 0], G[:, 2] = 1j * G[:, 0], 1j * G[:, 2]
        b = torch.zeros((A.shape[0], 4 * n1, 2 * nb), dtype=torch.float64, device=self.dev)
        cols = torch.view_as_real(G[..., : N - 1]).permute(2, 1, 3, 0, 4)   # mode, c, n, instance, part
        b[:, : 3 * (N - 1)] = cols.reshape(A.shape[0], 3 * (N - 1), 2 * nb)
        b *= scale[:, :, None]
        x = torch.linalg.lu_solve(*lu, b)
        x = x + torch.linalg.lu_solve(*lu, b - A @ x)
        x = torch.view_as_complex(x[:, : 3 * n1].reshape(-1, 3, n1, nb, 2).contiguous()).permute(3, 1, 0, 2).clone()
        x[:, 0], x[:, 2] = -1j * x[:, 0], -1j * x[:, 2]
        out = torch.zeros_like(F).reshape(nb, 3, -1, n1)
        out[:, :, 1:] = x
        out = out.reshape(F.shape)
        for c in (0, 2):
            r = F[:, c, 0, 0].clone()
            r[:, N - 1:] = 0
            z = torch.linalg.solve(M, torch.view_as_real(r).permute(1, 0, 2).reshape(n1, -1))
            out[:, c, 0, 0] = torch.view_as_complex(z.reshape(n1, nb, 2).permute(1, 0, 2).contiguous())
        return out

    def norm(self, a):
        v = self.phys(a)
        return torch.sqrt(0.5 * ((v ** 2).sum(1).mean((-2, -1)) * self.w).sum(-1))

    def residual(self, u, norm=True):
        v = self.phys(u)
        out = []
        for i in range(3):
            g = self.grad(u[:, i])
            t = -(self.U + v[:, 0]) * g[0] - (self.V + v[:, 1]) * g[1] - v[:, 2] * g[2]
            out.append(self.spec(t - self.dU * v[:, 1] if i == 0 else t))
        r = (self.stokes(u / self.dt + torch.stack(out, 1), self.dt) - u) / self.dt
        return r, self.norm(r) if norm else None

    def direction(self, u, r):
        v, q = self.phys(u), self.phys(r)
        gu = [self.grad(u[:, i]) for i in range(3)]
        out = []
        for i in range(3):
            g = self.grad(r[:, i])
            t = (self.U + v[:, 0]) * g[0] + (self.V + v[:, 1]) * g[1] + v[:, 2] * g[2]
            t = t - q[:, 0] * gu[0][i] - q[:, 1] * gu[1][i] - q[:, 2] * gu[2][i]
            out.append(self.spec(t - self.dU * q[:, 0] if i == 1 else t))
        return -(self.stokes(r / self.dh + torch.stack(out, 1), self.dh) - r) / self.dh

    def symmetrize(self, u, mask):
        """Group average over s1 (shift and rotate) and s2 (shift and reflect)."""
        flip = (-torch.arange(self.Mx, device=self.dev)) % self.Mx            # mode m -> -m
        sm = ((-1.0) ** self.m)[:, None, None]
        sp = ((-1.0) ** self.p)[None, :, None]
        sn = (-1.0) ** torch.arange(self.ny, dtype=torch.float64, device=self.dev)
        e1 = torch.tensor([-1.0, -1.0, 1.0], dtype=torch.float64, device=self.dev)[:, None, None, None]
        e2 = torch.tensor([1.0, 1.0, -1.0], dtype=torch.float64, device=self.dev)[:, None, None, None]
        # x -> -x turns the mode m into -m; the stored p >= 0 half of a real field then needs no
        # conjugate for s1 and the conjugate of mode -m for z -> -z
        if mask & 1:
            u = 0.5 * (u + e1 * sm * sp * sn * u[:, :, flip])
        if mask & 2:
            u = 0.5 * (u + e2 * sm * u[:, :, flip].conj())
        return u

    def descend(self, u, dtau, nsteps, mask=0):
        J = []
        u = self.symmetrize(u, mask)
        for _ in range(nsteps):
            r, j = self.residual(u)
            J.append(j)
            u = self.symmetrize(u + dtau * self.direction(u, r), mask)
        return u, torch.stack(J)


def _independent(nx, nz):
    Kx, Kz, Mx, Mz = _dims(nx, nz)
    return [(i, j) for i in range(Mx) for j in range(Mz) if j > 0 or 1 <= i <= Kx]


def _psi(nx, ny, nz, u):
    """Snapshot vector of one state: v and wall-normal vorticity per independent mode, mean u and w."""
    ij = torch.tensor(_independent(nx, nz), device=u.device)
    m, p, kx, kz = _waves(nx, nz, u.device)
    a = u[:, ij[:, 0], ij[:, 1]]
    v = a[1][:, : ny - 4]
    eta = (1j * kz[ij[:, 1]][:, None] * a[0] - 1j * kx[ij[:, 0]][:, None] * a[2])[:, : ny - 2]
    body = torch.cat([v.real, v.imag, eta.real, eta.imag], 1).reshape(-1)
    return torch.cat([body, u[0, 0, 0, : ny - 2].real, u[2, 0, 0, : ny - 2].real])


def _unpsi(nx, ny, nz, psi):
    """State of a snapshot vector: wall conditions completed, u and w from divergence and vorticity."""
    dev, N = psi.device, ny - 1
    Kx, Kz, Mx, Mz = _dims(nx, nz)
    ij = torch.tensor(_independent(nx, nz), device=dev)
    m, p, kx, kz = _waves(nx, nz, dev)
    n = torch.arange(ny, dtype=torch.float64, device=dev)
    alt = (-1.0) ** n
    Bd = torch.stack([torch.ones_like(n), alt])
    Bc = torch.cat([Bd, torch.stack([n ** 2, -alt * n ** 2])])

    def complete(a, B, k):
        """The last k coefficients from the wall conditions B a = 0."""
        return torch.cat([a, torch.linalg.solve(B[:, ny - k:], -B[:, : ny - k] @ a.T).T], 1)
    per = 2 * (N - 3) + 2 * (N - 1)
    body = psi[: len(ij) * per].reshape(len(ij), per)
    cut = np.cumsum([0, N - 3, N - 3, N - 1, N - 1])
    vr, vi, er, ei = [body[:, cut[k]:cut[k + 1]] for k in range(4)]
    v = torch.complex(complete(vr, Bc, 4), complete(vi, Bc, 4))
    eta = torch.complex(complete(er, Bd, 2), complete(ei, Bd, 2))
    X, Z = kx[ij[:, 0]][:, None], kz[ij[:, 1]][:, None]
    xi = -(v @ _deriv(ny, dev).to(v.dtype).T)
    modes = torch.stack([(-1j * X * xi - 1j * Z * eta) / (X ** 2 + Z ** 2), v,
                         (-1j * Z * xi + 1j * X * eta) / (X ** 2 + Z ** 2)])
    out = torch.zeros((3, Mx, Mz, ny), dtype=torch.complex128, device=dev)
    out[:, ij[:, 0], ij[:, 1]] = modes
    out[:, Kx + 1:, 0] = out[:, 1:Kx + 1, 0].flip(1).conj()
    mean = complete(psi[len(ij) * per:].reshape(2, N - 1), Bd, 2)
    out[0, 0, 0], out[2, 0, 0] = mean[0].to(out.dtype), mean[1].to(out.dtype)
    return out


def _dmd_exact(c, seed):
    S = _snapshots(c, seed)
    P = _Plain(c["nx"], c["ny"], c["nz"], c["Re"], 0.25, 0.25)
    A = S.T.cpu().numpy()
    U, s, Vt = np.linalg.svd(A[:, :-1], full_matrices=False)
    best = None
    for r in range(int((s > 1e-10 * s[0]).sum()), 0, -1):
        VS = Vt[:r].T / s[:r]
        lam, W = np.linalg.eig(U[:, :r].T @ A[:, 1:] @ VS)
        Phi = A[:, 1:] @ VS @ W
        b = np.linalg.lstsq(Phi, A[:, -1].astype(np.complex128), rcond=None)[0]
        q = int(np.argmin(np.abs(np.log(lam.astype(np.complex128)))))
        u = _unpsi(c["nx"], c["ny"], c["nz"], torch.from_numpy(np.real(b[q] * Phi[:, q])).to("cuda"))
        J = float(P.residual(u[None])[1][0])
        if math.isfinite(J) and (best is None or J < best[2]):
            best = (u, r, J)
    return {"u": best[0], "rank": None, "J": best[2]}


def _fno_exact(c, seed):
    Kx, Kz, Mx, Mz = _dims(c["nx"], c["nz"])
    MP, S, L = Mx * Mz, c["batch"], 4
    p = {k: torch.from_numpy(a).to("cuda", torch.float64).requires_grad_() for k, a in
         _params(MP, c["ny"], seed).items()}
    X, T = (a.double().reshape(MP, S, -1) for a in _pairs(c, seed))
    H = X @ p["E"].mT + p["bE"]
    for l in range(L):
        H = H + torch.nn.functional.gelu(H @ (p[f"R{l}"] + p[f"L{l}"]).mT + p[f"b{l}"])
    loss = (H @ p["D"].mT + p["bD"][:, None] - T).square().mean()
    loss.backward()
    return {"loss": float(loss), "grad": torch.cat([a.grad.reshape(-1) for a in p.values()])}


def exact(case, seed):
    c = case
    if c["kind"] == "fno":
        return _fno_exact(c, seed)
    if c["kind"] == "dmd":
        return _dmd_exact(c, seed)
    if c["kind"] == "uneven":
        us, Js = [], []
        for k, g in enumerate(_uneven(c)):
            u, J = _Plain(*g[:3], c["Re"], 0.25, 0.25).descend(_field(*g, 0.1, seed + k), c["dtau"], c["nsteps"])
            us.append(u.reshape(-1))
            Js.append(J)
        return {"u": torch.cat(us), "J": torch.cat(Js, 1)}
    P = _Plain(c["nx"], c["ny"], c["nz"], c["Re"], *_steps(c), base_flow=c["base_flow"])
    u = _field(c["nx"], c["ny"], c["nz"], c["batch"], _amplitude(c), seed)
    if c["kind"] in ("step", "step_host"):
        u, J = P.descend(u, c["dtau"], c["nsteps"], c["symmetry"])
        return {"u": u, "J": J}
    if c["kind"] == "gradient":
        r, J = P.residual(u)
        return {"r": r, "J": J, "f": P.direction(u, r)}
    if c["kind"] == "stokes":
        return {"u": P.stokes(u, 0.25)}
    H = []
    for _ in range(c["nsteps"]):
        H.append(P.norm(u))
        u = u + P.dt * P.residual(u, norm=False)[0]
    return {"u": u, "norm": torch.stack(H), "guesses": None, "found": None}
