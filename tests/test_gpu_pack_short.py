"""Weight pack of short one-group rows on both sides of the staged kernel's rule; every
byte and scale equals the oracle's (no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import soniq
    if not torch.cuda.is_available():
        pytest.skip("no CUDA GPU")
    return soniq


@pytest.mark.parametrize("N", [1, 192, 193])
@pytest.mark.parametrize("K,taps,pad", [(1, 1, 128), (3, 1, 128), (128, 1, 128), (14, 9, 32)])
@pytest.mark.parametrize("low,mode", [(True, "row"), (False, "row"), (False, "tensor")])
def test_short_rows(sq, N, K, taps, pad, low, mode):
    rng = np.random.default_rng(N + K)
    W = (rng.standard_normal((N, taps, K)) * 0.05).astype(np.float32)
    W[0, 0, 0] = np.nan
    W = W if taps > 1 else W[:, 0]
    perm, count, bits = rng.permutation(K).astype(np.int32), [K, 0] if low else [0, K], [3, 8]
    lay = sq.Layout(perm, count, bits, pad_unit=pad)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(W).cuda(), mode)
    assert sq.sync_status() == 0
    s_ref = oracle.weight_scales(W, perm, count, per_row=mode == "row")
    J = oracle.weight_codes(W, perm, count, bits, s_ref)
    assert np.array_equal(s_w.cpu().numpy(), s_ref)
    assert np.array_equal(Wp.cpu().numpy(), oracle.pack_weight_rows(J, count, bits, pad))
