"""Activation quantize under given scales: a few long rows cost less than with the
scales to be found per row (the same kernel and bytes, without the maxima)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


@pytest.mark.parametrize("M,K", [(1, 16384), (200, 8192), (400, 11008)])
def test_given_scales_cost_less_than_row_scales(sq, M, K):
    lay = sq.Layout(np.arange(K, dtype=np.int32), [K - K // 4, K // 4], [4, 8])
    A = torch.randn(M, K, device="cuda").half()
    Ap = torch.empty(M, lay.row_bytes(), dtype=torch.uint8, device="cuda")
    best = {}
    for mode in ("calibrated", "row"):
        s = torch.full((M, 2) if mode == "row" else (2,), 3.0, device="cuda")
        sq.quantize_act(lay, A, mode, s_a=s, Ap=Ap)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                sq.quantize_act(lay, A, mode, s_a=s, Ap=Ap)
        best[mode] = float("inf")
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            best[mode] = min(best[mode], a.elapsed_time(b))
    assert best["calibrated"] < best["row"], best
