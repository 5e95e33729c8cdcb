"""The fused per-mode network kernel (k_fno_mode) at the sizes where its tiling can go wrong:
sample counts around its 32-sample chunks, input widths that are not multiples of 16, every
width it serves, and a size it leaves to the separate products.  Against the FP64 reference
with the tolerances of the network's other tests (BF16 operands, 2^-9 relative each, through
the layers: 2e-2 forward, 5e-2 per gradient block); a train step must move the weights along
the gradient that loss_grad returns."""
import numpy as np
import pytest

from oracle import fno as ofno

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("MP,NY,W,L,S", [(3, 17, 32, 4, 1), (3, 17, 32, 4, 33), (2, 9, 16, 1, 32), (2, 11, 48, 2, 70),
                                         (2, 13, 64, 3, 31), (2, 65, 32, 4, 5), (2, 9, 24, 2, 40)])
def test_fused_network(pcf, MP, NY, W, L, S):
    rng = np.random.default_rng(MP + NY + W + S)
    net = pcf.FNO(MP, NY, width=W, layers=L, seed=0)
    p = ofno.init_params(MP, NY, W=W, L=L, seed=3)
    p["D"] = rng.standard_normal(p["D"].shape) / np.sqrt(W)
    p["bE"] = 0.1 * rng.standard_normal(W)
    p["bD"] = 0.1 * rng.standard_normal(p["bD"].shape)
    for l in range(L):
        p[f"b{l}"] = 0.1 * rng.standard_normal(W)
    net.set_params(net.pack(p))
    X, T = rng.standard_normal((MP, S, NY, 4)), rng.standard_normal((MP, S, NY, 4))
    Xd, Td = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (X, T))
    Yr, _ = ofno.forward(p, X, L)
    assert np.linalg.norm(net.forward(Xd).cpu().numpy() - Yr) <= 2e-2 * np.linalg.norm(Yr)
    loss, g = net.loss_grad(Xd, Td)
    lr, gr = ofno.loss_and_grads(p, X, T, L)
    assert abs(loss - lr) <= 2e-2 * lr
    g = g.cpu().numpy()
    gg = net.unpack(g)
    for k in gr:
        assert np.linalg.norm(gg[k] - gr[k]) <= 5e-2 * max(np.linalg.norm(gr[k]), 1e-30), k
    w0 = net.get_params()
    assert net.train_step(Xd, Td, 1e-3) == loss
    moved = net.get_params() - w0  # Adam's first step: -lr sign(g) where g is well above its epsilon
    big = np.abs(g) > 1e-5
    assert np.all(np.sign(moved[big]) == -np.sign(g[big]))
