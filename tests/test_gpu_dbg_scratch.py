"""A small call with debug accumulators takes the fused kernel, whatever scratch it is
given: the staged epilogue that writes them is slow."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


def test_small_call_with_debug_accumulators_leaves_its_scratch(sq):
    M, K, N = 200, 1024, 320
    d = wl.random_linear(4, M, K, N, 4, 8, 0.25)
    lay = sq.Layout(d["perm"], d["count"], d["bits"])
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda())
    need = sq.lib().soniq_mp_gemm_scratch_bytes(lay.ref, M, N, 0)
    assert need > 0
    buf = torch.full((need,), 7, dtype=torch.uint8, device="cuda")
    Y = torch.empty((M, N), dtype=torch.float16, device="cuda")
    acc = torch.empty((2, M, N), dtype=torch.int32, device="cuda")
    for dbg in (acc, None):
        assert sq.lib().soniq_mp_gemm(lay.ref, Ap.data_ptr(), s_a.data_ptr(), 0, M, Wp.data_ptr(), s_w.data_ptr(), N,
                                      Y.data_ptr(), 0, None if dbg is None else dbg.data_ptr(), 0, buf.data_ptr(), need, None,
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert sq.sync_status() == 0
        assert bool((buf == 7).all()) == (dbg is not None)
