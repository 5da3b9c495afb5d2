"""Layout variants quantized from staged rows by items of a chunk and some of a
tile's rows: tiles whose rows are split among warps, tiles of one and of many rows,
inputs off the 16-byte grid, calibrated scales on either side of the plain kernel's
rule; scales and bytes equal the oracle's (no tolerance).  And a layout without scale
runs costs about what one with runs does."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


def _at(x, offset):
    """x on the GPU, `offset` elements past an aligned address."""
    t = torch.from_numpy(x).cuda()
    buf = torch.zeros(t.numel() + offset, dtype=t.dtype, device="cuda")
    view = buf[offset:].view(t.shape)
    view.copy_(t)
    return view


def _check(sq, M, K, sub_k, kind, bits, mode, frac, offset):
    rng = np.random.default_rng(M + 7 * K + sub_k + offset)
    perm, count, _ = wl.assignment(rng, K, frac, 0)
    lay = sq.Layout(perm, count, list(bits), sub_k=sub_k, act_kind=kind)
    A = rng.standard_normal((M, K)).astype(np.float16)
    A[M // 2, ::11] = np.nan
    sa = np.asarray(oracle.sub_scales(A.astype(np.float32), perm, count, sub_k, mode == "row"), np.float32)
    given = None
    if mode == "calibrated":
        sa = sa * np.float32(0.8)
        given = torch.from_numpy(sa).cuda().reshape(lay.scale_shape(None))
    Ap, s_a = sq.quantize_act(lay, _at(A, offset), mode, s_a=given)
    W = (rng.standard_normal((M, K)) * 0.02).astype(np.float32)
    Wp, s_w = sq.pack_weights(lay, _at(W, offset))
    assert sq.sync_status() == 0
    sw = np.asarray(oracle.sub_scales(W, perm, count, sub_k, True), np.float32)
    wkind = [2 if k == 2 else 1 for k in kind]
    for X, s, per_row, kd, got_s, got in ((A.astype(np.float32), sa, mode == "row", kind, s_a, Ap),
                                          (W, sw, True, wkind, s_w, Wp)):
        U = oracle.codes_variant(X, perm, count, list(bits), kd, sub_k, s, per_row)
        assert np.array_equal(got_s.cpu().numpy().reshape(-1), s.reshape(-1))
        ref = oracle.pack_act_rows(oracle.code_patterns(U, count, list(bits), kd), count, list(bits), 128)
        assert np.array_equal(got.cpu().numpy(), ref)


@pytest.mark.parametrize("mode", ["row", "tensor", "calibrated"])
@pytest.mark.parametrize("M,K,sub_k,kind,bits,frac", [
    (5000, 100, 0, (1, 1), (4, 8), 0.3),         # two chunks: eight-fold split, many rows per tile
    (2500, 128, 0, (1, 1), (4, 4), 0.0),         # one chunk, one group
    (700, 700, 0, (2, 1), (1, 8), 0.25),         # uneven split
    (65, 2100, 128, (0, 1), (3, 6), 0.2),        # more chunks than warps by one or two
    (64, 2048, 0, (1, 1), (4, 8), 0.25), (65, 2047, 0, (1, 1), (5, 2), 1.0),
    (1, 4100, 256, (1, 0), (4, 8), 0.25), (640, 8200, 2048, (1, 1), (7, 8), 0.5)])
@pytest.mark.parametrize("offset", [0, 1])
def test_codes_and_scales(sq, M, K, sub_k, kind, bits, mode, frac, offset):
    _check(sq, M, K, sub_k, kind, bits, mode, frac, offset)


@pytest.mark.parametrize("mode", ["row", "tensor"])
def test_no_runs_costs_like_runs(sq, mode):
    """The same bytes and codes with one scale per group as with 128-code runs; a row's
    work spread over the CTA either way."""
    K, times = 4096, []
    A = torch.randn(16, K, device="cuda").half()
    for sub_k in (0, 128):
        lay = sq.Layout(np.arange(K, dtype=np.int32), [3072, 1024], [4, 8], sub_k=sub_k, act_kind=(1, 1))
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                sq.quantize_act(lay, A, mode)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[0] < 2 * times[1], times
