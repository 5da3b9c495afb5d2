"""Per-tensor quantize that streams its rows twice around a grid barrier: row
counts at its tile and ring edges, narrow and long rows, one- and two-group
layouts, scales outside the fast quotient's range, non-finite inputs; bytes and
scales equal the oracle's (no tolerance)."""
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


def _check(sq, M, K, bits, frac, pad_unit=128, scale=1.0, special=False):
    rng = np.random.default_rng(M + K)
    perm, count, _ = wl.assignment(rng, K, frac, 0)
    A = (rng.standard_normal((M, K)) * scale).astype(np.float16)
    if special:
        A[M // 2, ::7] = np.nan
        A[M - 1, 3] = -np.inf if special == "inf" else 0.0
    lay = sq.Layout(perm, count, list(bits), pad_unit=pad_unit)
    for _ in range(2):      # twice in a row: the barrier starts afresh
        Ap, s_a = sq.quantize_act(lay, torch.from_numpy(A).cuda())
    assert sq.sync_status() == 0
    s_ref = oracle.act_scales(A, perm, count)
    U = oracle.act_codes(A, perm, count, list(bits), s_ref)
    assert np.array_equal(s_a.cpu().numpy(), s_ref)
    assert np.array_equal(Ap.cpu().numpy(), oracle.pack_act_rows(U, count, list(bits), pad_unit))


@pytest.mark.parametrize("M", [304, 305, 1216, 1217, 2433, 6081])
@pytest.mark.parametrize("K,bits,frac", [(512, (4, 8), 0.25), (776, (2, 8), 0.2), (2048, (3, 6), 0.0)])
def test_row_counts(sq, M, K, bits, frac):
    _check(sq, M, K, bits, frac)


@pytest.mark.parametrize("M,K", [(400, 4096), (310, 11008), (305, 24992), (306, 32768)])
def test_row_lengths(sq, M, K):
    _check(sq, M, K, (1, 7), 0.5, pad_unit=32)


@pytest.mark.parametrize("scale,special", [(1.0, "nan"), (1.0, "inf"), (0.0, False), (6e-8, False)])
def test_special_values(sq, scale, special):
    _check(sq, 700, 1024, (4, 8), 1.0 if special == "nan" else 0.3, scale=scale, special=special)
