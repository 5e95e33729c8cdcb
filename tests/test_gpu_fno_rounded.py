"""The learned proposal's network against a reference that rounds where the kernels round: every product
takes BF16 operands, sums exactly and is rounded to FP32, everything else is FP32.  This leaves only the
order of FP32 sums, so that an element dropped at a tile's edge or a chunk's carry shows.

Tolerance: an FP32 difference of 2^-22 turns one BF16 rounding in about 10^4 by 2^-8, 4e-5 of a block's
norm; 1e-3 for blocks of few elements."""
import numpy as np
import pytest

from oracle import fno as ofno

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bf(a):
    return a.to(torch.bfloat16).double()


def _mm(a, b):
    return (_bf(a) @ _bf(b)).float()


def _reference(p, X, T, L):
    d = {k: torch.tensor(v, dtype=torch.float32, device="cuda") for k, v in p.items()}
    MP, S = X.shape[:2]
    Xf, Tf = X.reshape(MP, S, -1), T.reshape(MP, S, -1)
    H, Hs, Zs = _mm(Xf, d["E"].mT) + d["bE"], [], []
    for l in range(L):
        Hs.append(H)
        Z = _mm(H, (d[f"R{l}"] + d[f"L{l}"]).mT) + d[f"b{l}"]
        Zs.append(Z)
        H = H + torch.nn.functional.gelu(Z)
    Y = _mm(H, d["D"].mT) + d["bD"][:, None]
    dY = (2.0 / Y.numel()) * (Y - Tf)
    g = {"D": _mm(dY.mT, H), "bD": dY.sum(1)}
    dH = _mm(dY, d["D"])
    for l in reversed(range(L)):
        z = Zs[l].double()
        df = 0.5 * (1 + torch.erf(z / 2 ** 0.5)) + z * torch.exp(-0.5 * z * z) / (2 * np.pi) ** 0.5
        dZ = (dH * df).float()
        g[f"b{l}"], g[f"R{l}"] = dZ.sum((0, 1)), _mm(dZ.mT, Hs[l])
        g[f"L{l}"] = g[f"R{l}"].sum(0)
        dH = dH + _mm(dZ, d[f"R{l}"] + d[f"L{l}"])
    g["E"], g["bE"] = _mm(dH.mT, Xf), dH.sum((0, 1))
    return Y.reshape(X.shape), float((Y - Tf).double().square().mean()), g


# the last two widths take the separate products
@pytest.mark.parametrize("MP,NY,W,L,S", [(3, 17, 32, 4, 1), (3, 17, 32, 4, 31), (3, 17, 32, 4, 33), (2, 11, 16, 2, 70),
                                         (2, 9, 48, 1, 32), (3, 17, 24, 4, 33), (2, 33, 64, 4, 40)])
def test_against_the_rounded_reference(MP, NY, W, L, S):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as pcf
    pcf.load_library()
    rng = np.random.default_rng(MP + NY + W + S)
    net = pcf.FNO(MP, NY, width=W, layers=L, seed=0)
    p = ofno.init_params(MP, NY, W=W, L=L, seed=3)
    p["D"] = rng.standard_normal(p["D"].shape) / np.sqrt(W)
    p["bE"], p["bD"] = 0.1 * rng.standard_normal(W), 0.1 * rng.standard_normal(p["bD"].shape)
    for l in range(L):
        p[f"b{l}"] = 0.1 * rng.standard_normal(W)
    net.set_params(net.pack(p))
    X, T = (torch.tensor(rng.standard_normal((MP, S, NY, 4)), dtype=torch.float32, device="cuda") for _ in range(2))
    Yr, lr, gr = _reference(p, X, T, L)
    assert float((net.forward(X) - Yr).norm() / Yr.norm()) <= 1e-3
    loss, g = net.loss_grad(X, T)
    assert abs(loss - lr) <= 1e-3 * lr
    g = net.unpack(g.cpu().numpy())
    for k, v in gr.items():
        v = v.cpu().numpy()
        assert np.linalg.norm(g[k] - v) <= 1e-3 * np.linalg.norm(v), k
