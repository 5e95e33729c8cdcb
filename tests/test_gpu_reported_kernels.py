"""What a context reports of its kernels keeps the meaning of ABI version 3: variant 3 is the fused
half-step kernel whoever chose it, variant 1 the caller's solve_kind 2, and the separate analysis and
synthesis report the instances their CTAs group (one)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,batch,variant", [(0, 1, 3), (4, 1, 3), (2, 1, 1), (3, 1, 2), (5, 1, 4), (0, 16, 2), (1, 1, 0)])
def test_variant_and_groups(kind, batch, variant):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_00165_gb300 as pcf
    pcf.load_library()
    s = pcf.Solver(32, 33, 32, batch=batch, solve_kind=kind)
    assert s.solve_variant() == variant
    c = s.split_config()
    assert c["group"] == (0 if kind == 1 else 1)
    assert (c["analysis_mode_tile"] > 0) == (c["synthesis_mode_tile"] > 0) == (variant in (2, 4))
    assert (c["solve_group"] > 0) == (variant == 2)
    s.close()
