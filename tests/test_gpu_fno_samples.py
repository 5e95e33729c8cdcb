"""The learned proposal's forward pass over many samples: the samples of one mode are shared out over
CTAs, which moves no bit (each row is one sample's alone), and few modes do not leave the GPU idle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("MP,S", [(1, 33), (2, 70), (45, 65), (45, 256), (200, 96), (400, 40)])
def test_rows_do_not_depend_on_their_number(pcf, MP, S):
    net = pcf.FNO(MP, 9, width=16, layers=2, seed=1)
    X = torch.randn((MP, S, 9, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(S))
    Y = net.forward(X)
    for k in {0, 31, 32, S - 1}:
        assert torch.equal(net.forward(X[:, k:k + 1].contiguous()), Y[:, k:k + 1])


def test_many_samples_of_few_modes(pcf):
    """45 modes: 32 times the samples take less than eight times as long (one CTA per mode: 13 times)."""
    net, times = pcf.FNO(45, 17, seed=0), []
    for S in (32, 1024):
        X = torch.randn((45, S, 17, 4), device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = np.inf
        for _ in range(8):
            a.record()
            for _ in range(5):
                net.forward(X)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] <= 8 * times[0]
