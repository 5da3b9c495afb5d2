"""Who owns the binding's scratch: captured calls get memory of their graph (the
quantize scratch zeroed within it), and the library asks for none where none is
read."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import build, soniq
    build.build()
    return soniq


@pytest.mark.parametrize("use", ["quantize", "gemm"])
def test_captured_scratch_is_not_cached(sq, use, monkeypatch):
    monkeypatch.setattr(sq, "_scratch", {})
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    bufs = [sq._get_scratch(4096, torch.device("cpu"), None, use) for _ in range(2)]
    assert bufs[0].data_ptr() != bufs[1].data_ptr() and not sq._scratch
    if use == "quantize":
        assert not any(b.any() for b in bufs)


@pytest.mark.parametrize("M,K,need", [(1, 16384, False), (64, 256, False), (1, 16385, True), (65, 252, True),
                                      (64, 257, True)])
def test_quantize_scratch_size(sq, M, K, need):
    c = sq.CLayout()
    c.K, c.n_groups, c.pad_unit = K, 1, 128
    c.count[0], c.bits_w[0], c.bits_a[0] = K, 4, 4
    assert (sq.lib().soniq_quantize_act_scratch_bytes(ctypes.byref(c), M, 0) > 0) == need
    c.sub_k = 128
    assert sq.lib().soniq_quantize_act_scratch_bytes(ctypes.byref(c), M, 0) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("own_stream", [False, True])
def test_graphs_with_per_tensor_quantize(sq, own_stream):
    """Graphs captured on one stream that has not quantized before: replayed second one
    first, then side by side; every replay gives the oracle's scales and bytes."""
    calls = []
    for seed, (M, K) in enumerate([(64, 512), (1280, 5000), (3, 40), (70, 234)]):   # one pass, streamed, one CTA, scalar rows
        rng = np.random.default_rng(seed)
        perm, count, _ = wl.assignment(rng, K, 0.25, 0)
        A = rng.standard_normal((M, K)).astype(np.float16)
        s_ref = oracle.act_scales(A, perm, count)
        U = oracle.act_codes(A, perm, count, [4, 8], s_ref)
        lay = sq.Layout(perm, count, [4, 8])
        calls.append((lay, torch.from_numpy(A).cuda(), s_ref, oracle.pack_act_rows(U, count, [4, 8], 128),
                      torch.zeros(2, device="cuda"), torch.zeros(M, lay.row_bytes(), dtype=torch.uint8, device="cuda")))
    capture = torch.cuda.Stream()
    arg = torch.cuda.Stream() if own_stream else None      # the call's own stream, forked from the capturing one
    graphs = []
    for lay, A, _, _, s, Ap in calls:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=capture):
            if own_stream:
                arg.wait_stream(capture)
            sq.quantize_act(lay, A, s_a=s, Ap=Ap, stream=arg)
            sq.quantize_act(lay, A, s_a=s, Ap=Ap, stream=arg)
            if own_stream:
                capture.wait_stream(arg)
        graphs.append(g)

    def check():
        torch.cuda.synchronize()
        assert sq.sync_status() == 0
        for _, _, s_ref, ref, s, Ap in calls:
            assert np.array_equal(s.cpu().numpy(), s_ref) and np.array_equal(Ap.cpu().numpy(), ref)
            s.zero_()
            Ap.zero_()

    for g in reversed(graphs):
        g.replay()
    check()
    streams = [torch.cuda.Stream() for _ in graphs]
    for _ in range(20):
        for g, st in zip(graphs, streams):
            with torch.cuda.stream(st):
                g.replay()
    check()
