"""Next-layer codes of a layer whose group is accumulated in exact segments: codes and
outputs equal those of the general epilogue bit for bit, with and without outputs, row
scales, one and two groups, scales outside the fast quotient's range."""
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


def _both(sq, call, lay2, s2, M):
    """(codes, outputs) of the general epilogue (debug accumulators) and of the segmented one."""
    out = []
    for dbg in (True, False):
        nxt = sq.NextLayer(lay2, torch.tensor(s2, device="cuda"), M=M)
        Y = call(nxt, dbg, True)
        out.append((nxt.Ap, Y.view(torch.int16)))
    nxt = sq.NextLayer(lay2, torch.tensor(s2, device="cuda"), M=M)
    call(nxt, False, False)
    assert sq.sync_status() == 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[0][0], nxt.Ap)
    assert out[0][0].any()


@pytest.mark.parametrize("M,K,N,bits,frac", [(14, 2100, 128, (8, 8), 0.0), (253, 1856, 640, (4, 8), 0.7),
                                             (1270, 6032, 128, (6, 7), 1.0), (300, 1500, 4224, (8, 3), 0.1)])
@pytest.mark.parametrize("mode", ["tensor", "row"])
@pytest.mark.parametrize("s2", [(40.0, 60.0), (1e-25, 30.0)])
def test_linear(sq, M, K, N, bits, frac, mode, s2):
    d = wl.random_linear(M + K, M, K, N, bits[0], bits[1], frac)
    lay = sq.Layout(d["perm"], d["count"], d["bits"])
    n1 = N // 256 * 128
    lay2 = sq.Layout(np.arange(N, dtype=np.int32), [N - n1, n1], [3, 8])
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda() * 30)
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda(), mode)
    acc = torch.empty((2, M, N), dtype=torch.int32, device="cuda")
    _both(sq, lambda nxt, dbg, wy: sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode, acc_dbg=acc if dbg else None, next=nxt,
                                              write_y=wy), lay2, s2, M)


def test_conv(sq):
    c = wl.make_conv(wl.ConvSpec("seg", batch=2, H=9, W=11, C=256, C_out=256, R=3, S=3, stride=(1, 1), pad=(1, 1),
                                 bits_lo=4, bits_hi=8, frac_hi=0.6, seed=3))
    lay = sq.Layout(c["perm"], c["count"], c["bits"], pad_unit=32)
    lay2 = sq.Layout(np.arange(256, dtype=np.int32), [128, 128], [4, 8], pad_unit=32)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(c["W"]).cuda())
    Xp, s_a = sq.quantize_act(lay, torch.from_numpy(c["X"]).cuda().reshape(-1, 256))
    M = 2 * 9 * 11
    acc = torch.empty((2, M, 256), dtype=torch.int32, device="cuda")
    cd = sq.conv_desc(2, 9, 11, 256)
    _both(sq, lambda nxt, dbg, wy: sq.mp_conv2d(lay, cd, Xp, s_a, Wp, s_w, acc_dbg=acc if dbg else None, next=nxt,
                                                write_y=wy), lay2, (0.5, 0.8), M)
