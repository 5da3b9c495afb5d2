"""Small calls that take the staged path with scratch: scratch off its alignment
leaves them on the fused kernel (an error where only the staged path will do),
and captured calls use memory of their graph.  Outputs are equal bit for bit."""
import ctypes

import numpy as np
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


def _layer(sq, M, K, N, seed):
    rng = np.random.default_rng(seed)
    perm, count, _ = wl.assignment(rng, K, 0.25, 0)
    lay = sq.Layout(perm, count, [4, 8])
    W = torch.from_numpy(rng.standard_normal((N, K)).astype(np.float32)).cuda()
    A = torch.from_numpy(rng.standard_normal((M, K)).astype(np.float16)).cuda()
    return lay, sq.quantize_act(lay, A, "row"), sq.pack_weights(lay, W)


@pytest.mark.parametrize("offset", [16, 4, 1])
def test_misaligned_scratch_is_not_used_by_small_calls(sq, offset):
    M, K, N = 64, 512, 192
    lay, (Ap, s_a), (Wp, s_w) = _layer(sq, M, K, N, 1)
    ref = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, scale_mode="row", flags=sq.FLAG_FORCE_FUSED)
    need = sq.lib().soniq_mp_gemm_scratch_bytes(lay.ref, M, N, 0)
    assert need > 0
    buf = torch.full((need + 512,), 7, dtype=torch.uint8, device="cuda")
    Y = torch.empty_like(ref)

    def call(flags):
        return sq.lib().soniq_mp_gemm(lay.ref, Ap.data_ptr(), s_a.data_ptr(), 1, M, Wp.data_ptr(), s_w.data_ptr(), N,
                                      Y.data_ptr(), 0, None, flags, buf.data_ptr() + offset, need, None,
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    assert call(0) == 0
    assert sq.sync_status() == 0
    assert torch.equal(Y, ref) and bool((buf == 7).all())
    assert call(sq.FLAG_FORCE_STAGED) == 3


def test_captured_calls_own_their_scratch(sq):
    layers = [_layer(sq, 64, 512, 192, 2), _layer(sq, 200, 1024, 320, 3)]
    refs = [sq.mp_gemm(l, *q, *w, scale_mode="row") for l, q, w in layers]
    graphs, outs = [], []
    for (l, q, w), r in zip(layers, refs):
        Y = torch.zeros_like(r)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sq.mp_gemm(l, *q, *w, Y=Y, scale_mode="row")
        graphs.append(g)
        outs.append(Y)
    streams = [torch.cuda.Stream() for _ in graphs]
    for _ in range(20):
        for g, s in zip(graphs, streams):
            with torch.cuda.stream(s):
                g.replay()
    torch.cuda.synchronize()
    assert sq.sync_status() == 0
    for y, r in zip(outs, refs):
        assert torch.equal(y, r)
