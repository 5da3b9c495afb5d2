"""Few activation rows on warp-level tensor instructions: row counts at its tile
edges, weight rows at the edges of its stages and of the SMs' shares, every
weight width, K at the ring and block-range edges, rows too long for it; codes
at their extremes.  Accumulators equal the oracle's, outputs lie within the fp16
tolerance of the other tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from helpers import assert_y_close  # noqa: E402
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


def _check(sq, d, bits_a=None, pad=128, mode="tensor"):
    bits_w = d["bits"]
    bits_a = bits_a or bits_w
    lay = sq.Layout(d["perm"], d["count"], bits_w, bits_a, pad_unit=pad)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda(), mode)
    M, N = d["A"].shape[0], d["W"].shape[0]
    acc = torch.full((2, M, N), -1, dtype=torch.int32, device="cuda")
    Y = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode, acc_dbg=acc)
    Y2 = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode)
    assert sq.sync_status() == 0
    assert torch.equal(Y.view(torch.int16), Y2.view(torch.int16))
    r = oracle.linear(d["A"], d["W"], d["perm"], d["count"], bits_a, bits_w, pad_unit=pad, act_mode=mode)
    got = acc.cpu().numpy().astype(np.int64)
    for g in range(2):
        if d["count"][g]:
            assert np.array_equal(got[g], r["acc"][g])
    terms = oracle.epilogue_terms(r["acc"], r["s_a"], r["s_w"], bits_a, bits_w, s_a_per_row=mode == "row")
    assert_y_close(Y.float().cpu().numpy(), r["Y64"].astype(np.float16), terms)


@pytest.mark.parametrize("M", [3, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("K,N,bits,frac", [(130, 1, (4, 8), 0.3), (512, 17, (2, 8), 0.25), (1000, 333, (3, 6), 0.15),
                                           (2048, 2433, (1, 7), 0.5), (600, 4880, (4, 5), 0.0), (300, 100, (1, 8), 1.0)])
def test_shapes(sq, M, K, N, bits, frac):
    _check(sq, wl.random_linear(M + K, M, K, N, bits[0], bits[1], frac))


@pytest.mark.parametrize("M,K,pad", [(5, 333, 32), (12, 4096, 32), (16, 8192, 128), (12, 20000, 128), (31, 6000, 128)])
def test_long_rows_and_pads(sq, M, K, pad):
    _check(sq, wl.random_linear(K, M, K, 200, 2, 6, 0.2), pad=pad, mode="row")


@pytest.mark.parametrize("bits_a,bits_w", [((8, 8), (8, 8)), ((4, 8), (8, 4)), ((8, 1), (1, 8))])
def test_extreme_codes(sq, bits_a, bits_w):
    """Every product at its largest over K = 4096: partial sums pass 2^24 many times."""
    M, K, N = 7, 4096, 40
    perm, count, _ = wl.assignment(np.random.default_rng(1), K, 0.5, 0)
    A = np.ones((M, K), np.float16)
    W = np.where(np.arange(N)[:, None] % 2 == 0, -1.0, 1.0).astype(np.float32) * np.ones((1, K), np.float32)
    _check(sq, dict(A=A, W=W, perm=perm, count=count, bits=list(bits_w)), bits_a=list(bits_a))
