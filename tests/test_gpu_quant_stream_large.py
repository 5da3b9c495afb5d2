"""The streamed per-tensor quantize at inputs that no other one-launch kernel takes
(rows beyond the grid's shared memory; one launch rules out the two passes): tiles per
CTA at and above the ring's stages, short last tiles, one row per tile, scales outside
the fast quotient's range, non-finite inputs, a lost grid-barrier arrival.  Bytes and
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


def _case(sq, M, K, bits, frac, pad, scale=1.0, special=None):
    rng = np.random.default_rng(M + K)
    perm, count, _ = wl.assignment(rng, K, frac, 0)
    A = (rng.standard_normal((M, K), dtype=np.float32) * scale).astype(np.float16)
    if special is not None:
        A[M // 2, ::7] = np.nan
        A[M - 1, 3] = special
    lay = sq.Layout(perm, count, list(bits), pad_unit=pad)
    # too large for the one-pass kernel, which holds each SM's share of the packed rows (fp16)
    # and the positions in 200 KB
    share = -(-M // torch.cuda.get_device_properties(0).multi_processor_count)
    assert share * (lay.group_codes(0) + lay.group_codes(1)) * 2 + 2 * K > 200 * 1024
    s_ref = oracle.act_scales(A, perm, count)
    U = oracle.act_codes(A, perm, count, list(bits), s_ref)
    return lay, torch.from_numpy(A).cuda(), s_ref, oracle.pack_act_rows(U, count, list(bits), pad)


def _check(sq, lay, A, s_ref, ref):
    before = sq.launch_count()
    Ap, s_a = sq.quantize_act(lay, A)
    assert sq.launch_count() == before + 1
    assert sq.sync_status() == 0
    assert np.array_equal(s_a.cpu().numpy(), s_ref)
    assert np.array_equal(Ap.cpu().numpy(), ref)


@pytest.mark.parametrize("M,K,bits,frac,pad", [
    (31009, 512, (4, 8), 0.25, 128), (17329, 776, (2, 8), 0.2, 128), (20001, 776, (3, 6), 0.2, 32),
    (7753, 2048, (3, 6), 0.0, 128), (3900, 4096, (4, 8), 0.25, 128), (4560, 4096, (1, 7), 1.0, 128),
    (1369, 11008, (5, 2), 0.5, 32), (913, 16384, (8, 4), 0.3, 32), (457, 24992, (4, 8), 0.5, 32)])
def test_shapes(sq, M, K, bits, frac, pad):
    case = _case(sq, M, K, bits, frac, pad)
    for _ in range(2):      # twice in a row: the barrier starts afresh
        _check(sq, *case)


@pytest.mark.parametrize("scale,special,frac", [(1.0, 0.0, 0.3), (1.0, -np.inf, 0.3), (1.0, np.inf, 1.0), (0.0, None, 0.3),
                                                (6e-8, None, 0.3)])
def test_special_values(sq, scale, special, frac):
    _check(sq, *_case(sq, 3953, 4096, (4, 8), frac, 128, scale, special))


def test_lost_arrival(sq):
    case = _case(sq, 3953, 4096, (4, 8), 0.25, 128)
    _check(sq, *case)
    sq.test_drop_barrier_arrival()
    sq.quantize_act(case[0], case[1])
    assert sq.sync_status() == 5            # SONIQ_ERR_TIMEOUT, then cleared and the scratch zeroed
    _check(sq, *case)
