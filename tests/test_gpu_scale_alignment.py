"""Scale arrays need 4-byte alignment and no more: arrays that begin on an odd
float (views into a flat buffer) give the bits of aligned ones, in every kernel
behind soniq_mp_gemm and soniq_mp_conv2d."""
import pytest

torch = pytest.importorskip("torch")
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
GEMV, FUSED, STAGED, SKINNY = 1, 2 | 4, 2 | 8, 16


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


def _odd(t):
    """t's values in memory that begins 4 bytes past an 8-byte boundary."""
    buf = torch.full((t.numel() + 3,), float("nan"), dtype=t.dtype, device=t.device)
    view = buf[1:1 + t.numel()].view(t.shape)
    view.copy_(t)
    assert view.data_ptr() % 8 == 4
    return view


@pytest.mark.parametrize("M,K,N,frac,flags,sub_k,dbg", [
    (300, 640, 320, 0.25, STAGED, 0, False), (2432, 200, 2047, 0.25, STAGED, 0, False),    # one piece per group
    (300, 2560, 480, 0.6, STAGED, 0, False), (2048, 2500, 513, 0.5, STAGED, 0, False),     # segments
    (130, 640, 320, 0.25, STAGED, 0, True), (130, 640, 320, 0.25, 0, 128, False),          # debug accumulators; runs
    (130, 640, 320, 0.25, FUSED, 0, False), (1, 640, 320, 0.25, GEMV, 0, False),
    (9, 640, 320, 0.25, 0, 0, False), (16, 640, 320, 0.25, SKINNY, 0, False)])
@pytest.mark.parametrize("mode", ["tensor", "row"])
def test_linear(sq, M, K, N, frac, flags, sub_k, dbg, mode):
    d = wl.random_linear(M + K, M, K, N, 4, 8, frac)
    lay = sq.Layout(d["perm"], d["count"], d["bits"], sub_k=sub_k)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda(), mode)
    acc = torch.empty((2, M, N), dtype=torch.int32, device="cuda") if dbg else None
    ref = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode, acc_dbg=acc, flags=flags)
    Y = sq.mp_gemm(lay, Ap, _odd(s_a), Wp, _odd(s_w), mode, acc_dbg=acc, flags=flags)
    assert sq.sync_status() == 0
    assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("flags", [STAGED, FUSED])
def test_conv(sq, flags):
    c = wl.make_conv(wl.ConvSpec("odd", batch=2, H=11, W=9, C=64, C_out=80, R=3, S=3, stride=(1, 1), pad=(1, 1),
                                 bits_lo=4, bits_hi=8, frac_hi=0.3, seed=1))
    lay = sq.Layout(c["perm"], c["count"], c["bits"], pad_unit=32)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(c["W"]).cuda())
    Xp, s_a = sq.quantize_act(lay, torch.from_numpy(c["X"]).cuda().reshape(-1, 64))
    cd = sq.conv_desc(2, 11, 9, 80)
    ref = sq.mp_conv2d(lay, cd, Xp, s_a, Wp, s_w, flags=flags)
    Y = sq.mp_conv2d(lay, cd, Xp, _odd(s_a), Wp, _odd(s_w), flags=flags)
    assert sq.sync_status() == 0
    assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("K,frac,conv", [(640, 0.25, False), (2560, 0.6, False), (64, 0.3, True)])
def test_next_layer(sq, K, frac, conv):
    N = 384
    lay2 = sq.Layout(list(range(N)), [256, 128], [4, 8])
    if conv:
        d = wl.make_conv(wl.ConvSpec("odd", batch=2, H=11, W=9, C=K, C_out=N, R=3, S=3, stride=(1, 1), pad=(1, 1),
                                     bits_lo=4, bits_hi=8, frac_hi=frac, seed=2))
        A = torch.from_numpy(d["X"]).cuda().reshape(-1, K)
    else:
        d = wl.random_linear(3, 300, K, N, 4, 8, frac)
        A = torch.from_numpy(d["A"]).cuda()
    lay = sq.Layout(d["perm"], d["count"], d["bits"], pad_unit=32 if conv else 128)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, A)
    out = []
    for f in (lambda t: t, _odd):
        nxt = sq.NextLayer(lay2, f(torch.tensor([0.7, 1.3], device="cuda")), M=A.shape[0])
        if conv:
            Y = sq.mp_conv2d(lay, sq.conv_desc(2, 11, 9, N), Ap, f(s_a), Wp, f(s_w), next=nxt)
        else:
            Y = sq.mp_gemm(lay, Ap, f(s_a), Wp, f(s_w), next=nxt)
        out.append((Y.view(torch.int16), nxt.Ap))
    assert sq.sync_status() == 0
    for a, b in zip(*out):
        assert torch.equal(a, b)
