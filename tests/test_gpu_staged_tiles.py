"""Tile widths and epilogues of the staged GEMM: shapes that take each of its
kernels (64-, 128- and 256-column tiles, CTA pairs, outputs by 64-byte batches or
TMA stores, segments, E2M1 layouts, scale runs), with ragged rows and columns.

The kernel's outputs equal the general epilogue's (debug accumulators) bit for
bit, and the accumulators equal the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_2311_14114_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
STAGED = 2 | 8


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


def _check(sq, M, K, N, bits, frac, mode, dtype, sub_k=0, kind=(0, 0)):
    d = wl.random_linear(M + K + N, M, K, N, bits[0], bits[1], frac, n_outliers=2)
    lay = sq.Layout(d["perm"], d["count"], d["bits"], sub_k=sub_k, act_kind=kind)
    A, W = torch.from_numpy(d["A"]).cuda(), torch.from_numpy(d["W"]).cuda()
    Wp, s_w = sq.pack_weights(lay, W)
    Ap, s_a = sq.quantize_act(lay, A, mode)
    shape = (2, lay.scale_runs(), M, N) if sub_k else (2, M, N)
    acc = torch.zeros(shape, dtype=torch.int32, device="cuda")
    # an output buffer inside guard values: nothing is written beyond it
    buf = torch.full((M * N + 64,), 7.0, dtype=dtype, device="cuda")
    Y = buf[32:32 + M * N].view(M, N)
    sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode, Y=Y, flags=0 if sub_k else STAGED)
    ref = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, mode, out_dtype=dtype, acc_dbg=acc, flags=0 if sub_k else STAGED)
    assert sq.sync_status() == 0
    assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))
    assert (buf[:32] == 7).all() and (buf[32 + M * N:] == 7).all()
    rows = np.unique(np.linspace(0, M - 1, min(M, 24)).astype(np.int64))
    if sub_k:
        r = oracle.linear_variant(d["A"], d["W"], d["perm"], d["count"], d["bits"], d["bits"], kind=kind, sub_k=sub_k,
                                  act_mode=mode, rows=rows)
    else:
        r = oracle.linear(d["A"], d["W"], d["perm"], d["count"], d["bits"], d["bits"], act_mode=mode, rows=rows)
    got = acc.cpu().numpy().astype(np.int64)[..., rows, :]
    assert np.array_equal(got, r["acc"].reshape(got.shape))


@pytest.mark.parametrize("M,K,N,bits,frac", [
    (1, 130, 1, (4, 8), 0.3), (40, 300, 72, (2, 8), 0.25), (129, 256, 65, (4, 8), 0.5),     # 64 columns, one wave
    (2000, 200, 1000, (4, 8), 0.3), (1999, 400, 1001, (3, 6), 0.2),                         # 128 columns
    (2432, 200, 2048, (4, 8), 0.25), (2431, 200, 2046, (4, 8), 0.25),                       # 256, TMA stores / N % 8
    (2432, 1600, 2040, (4, 8), 0.2),                                                        # 256, batches
    (2047, 2048, 2300, (4, 8), 0.25),                                                       # pairs, ragged
    (700, 2500, 520, (4, 8), 0.6), (2048, 2500, 2301, (4, 8), 0.5), (300, 2400, 70, (8, 4), 0.0),   # segments
    (300, 2560, 480, (2, 8), 0.2), (2100, 2304, 2397, (2, 2), 0.0), (900, 4000, 479, (2, 8), 0.4),  # E2M1
])
@pytest.mark.parametrize("mode,dtype", [("tensor", torch.float16), ("row", torch.bfloat16)])
def test_tiles(sq, M, K, N, bits, frac, mode, dtype):
    _check(sq, M, K, N, bits, frac, mode, dtype)


@pytest.mark.parametrize("M,K,N,sub_k", [(33, 300, 65, 128), (1001, 700, 1111, 256), (2048, 640, 1024, 128),
                                         (2500, 384, 2050, 128)])
@pytest.mark.parametrize("mode,kind", [("tensor", (0, 0)), ("row", (1, 1))])
def test_scale_runs(sq, M, K, N, sub_k, mode, kind):
    _check(sq, M, K, N, (4, 8), 0.3, mode, torch.float16, sub_k, kind)
