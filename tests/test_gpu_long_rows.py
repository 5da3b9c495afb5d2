"""Staged GEMM of long rows: packed rows that one, two, four and eight warps expand
together (and one CTA per SM at the longest), row counts that leave a tile short,
activation rows off the 16-byte grid.  Accumulators equal the oracle's; outputs equal
those of a fresh call with aligned rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu
STAGED = 2 | 8


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


@pytest.mark.parametrize("M,N,K,bits_a,bits_w,frac,pad", [
    (37, 67, 6900, (8, 8), (8, 8), 0.0, 128), (5, 130, 7000, (8, 8), (8, 8), 0.0, 128),
    (64, 64, 16000, (8, 4), (8, 4), 0.3, 128), (1, 9, 16001, (4, 8), (4, 8), 0.9, 128),
    (33, 301, 30000, (8, 8), (7, 8), 0.0, 128), (9, 1, 36032, (7, 7), (7, 7), 0.0, 32),
    (700, 35, 36032, (7, 7), (4, 4), 0.0, 32), (34, 66, 60000, (8, 2), (8, 3), 0.2, 128)])
@pytest.mark.parametrize("offset", [0, 4])
def test_long_rows(sq, M, N, K, bits_a, bits_w, frac, pad, offset):
    rng = np.random.default_rng(K + M)
    hi = int(frac * K)
    count = [K - hi, hi]
    U = np.concatenate([rng.integers(0, 1 << bits_a[g], (M, count[g])) for g in (0, 1)], axis=1).astype(np.uint8)
    J = np.concatenate([rng.integers(-(1 << (bits_w[g] - 1)), 1 << (bits_w[g] - 1), (N, count[g])) for g in (0, 1)],
                       axis=1).astype(np.int8)
    lay = sq.Layout(np.arange(K, dtype=np.int32), count, bits_w, bits_a, pad_unit=pad)
    packed = torch.from_numpy(oracle.pack_act_rows(U, count, list(bits_a), pad)).cuda()
    buf = torch.zeros(packed.numel() + offset, dtype=torch.uint8, device="cuda")
    Ap = buf[offset:].view(packed.shape)
    Ap.copy_(packed)
    Wp = torch.from_numpy(oracle.pack_weight_rows(J, count, list(bits_w), pad)).cuda()
    s_a = torch.tensor([1.0, 0.5], device="cuda")
    s_w = torch.rand(N, 2, device="cuda")
    acc = torch.full((2, M, N), -1, dtype=torch.int32, device="cuda")
    sq.mp_gemm(lay, Ap, s_a, Wp, s_w, acc_dbg=acc, flags=STAGED)
    Y = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, flags=STAGED)
    ref = sq.mp_gemm(lay, packed, s_a, Wp, s_w, flags=STAGED)
    assert sq.sync_status() == 0
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), oracle.gemm_acc(U, J, count))
    assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))
