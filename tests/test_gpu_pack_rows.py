"""Weight pack with bulk-staged rows: row lengths at the edges of its register
tiles, rows and tensors off the 16-byte grid, filter taps, one-group layouts and
the rows too long for it; bytes and scales equal the oracle's (no tolerance)."""
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


def _check(sq, K, taps, N, bits, frac, pad_unit, shift, mode, special=False):
    rng = np.random.default_rng(K + taps + N)
    perm, count, _ = wl.assignment(rng, K, frac, 0)
    W = (rng.standard_normal((N, taps, K)) * 0.05).astype(np.float32)
    if special:
        W[0] = 0.0
        W[1, 0, :: max(1, K // 5)] = np.nan
        W[2, -1, K // 2] = np.inf
        W[3] *= np.float32(1e-38)
    if taps == 1:
        W = W[:, 0]
    lay = sq.Layout(perm, count, list(bits), pad_unit=pad_unit)
    flat = torch.zeros(W.size + shift, dtype=torch.float32, device="cuda")
    Wd = flat[shift:].view(W.shape)
    Wd.copy_(torch.from_numpy(W))
    Wp, s_w = sq.pack_weights(lay, Wd, mode)
    assert sq.sync_status() == 0
    s_ref = oracle.weight_scales(W, perm, count, per_row=mode == "row")
    J = oracle.weight_codes(W, perm, count, list(bits), s_ref)
    assert np.array_equal(s_w.cpu().numpy(), s_ref)
    assert np.array_equal(Wp.cpu().numpy(), oracle.pack_weight_rows(J, count, list(bits), pad_unit))


# blocks per warp 4 | 8 | 16 | 24, the last row length each takes and the next; then rows beyond the kernel
@pytest.mark.parametrize("K", [1, 3, 127, 130, 896, 1024, 1026, 4096, 4353, 11008, 11777, 17408, 20001])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_row_lengths_and_alignment(sq, K, shift):
    _check(sq, K, 1, 5, (3, 6), 0.15, 128, shift, "row", special=K > 100)


@pytest.mark.parametrize("bits,frac", [((1, 8), 0.5), ((2, 7), 0.0), ((4, 5), 1.0)])
@pytest.mark.parametrize("mode", ["row", "tensor"])
def test_groups_and_scale_modes(sq, bits, frac, mode):
    _check(sq, 777, 1, 700, bits, frac, 128, 2, mode, special=mode == "row")


@pytest.mark.parametrize("K,taps,N", [(64, 9, 64), (77, 9, 400), (33, 25, 10), (512, 9, 33)])
def test_filter_taps(sq, K, taps, N):
    _check(sq, K, taps, N, (4, 8), 0.3, 32, 1, "row", special=True)
