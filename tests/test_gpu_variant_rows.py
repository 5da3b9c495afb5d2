"""Layout variants quantized from staged rows: tile heights, run lengths and
row ends at their edges, rows that fall back to the plain kernels; every packed
byte and scale equals the oracle's (no tolerance), weights and activations."""
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


@pytest.mark.parametrize("M,K", [(1, 128), (9, 1000), (17, 2047), (33, 3001), (20, 13000), (3, 30000)])
@pytest.mark.parametrize("sub_k,kind,bits", [(128, (1, 1), (4, 8)), (256, (0, 1), (2, 6)), (640, (2, 0), (1, 3)),
                                             (0, (1, 2), (5, 1))])
@pytest.mark.parametrize("mode", ["row", "tensor"])
def test_codes_and_scales(sq, M, K, sub_k, kind, bits, mode):
    rng = np.random.default_rng(M + K + sub_k)
    perm, count, _ = wl.assignment(rng, K, 0.3, 0)
    A = rng.standard_normal((M, K)).astype(np.float16)
    W = (rng.standard_normal((M, K)) * 0.02).astype(np.float32)
    if K > 500:
        A[M // 2, ::11] = np.nan
        W[M - 1, 3::13] = 0.0
    lay = sq.Layout(perm, count, list(bits), sub_k=sub_k, act_kind=kind)
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(A).cuda(), mode)
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(W).cuda())
    assert sq.sync_status() == 0
    A32 = A.astype(np.float32)
    sa_ref = oracle.sub_scales(A32, perm, count, sub_k, mode == "row")
    U = oracle.codes_variant(A32, perm, count, list(bits), kind, sub_k, sa_ref, mode == "row")
    assert np.array_equal(s_a.cpu().numpy().reshape(-1), np.asarray(sa_ref, np.float32).reshape(-1))
    ref = oracle.pack_act_rows(oracle.code_patterns(U, count, list(bits), kind), count, list(bits), 128)
    assert np.array_equal(Ap.cpu().numpy(), ref)
    sw_ref = oracle.sub_scales(W, perm, count, sub_k, True)
    wkind = [2 if k == 2 else 1 for k in kind]
    J = oracle.codes_variant(W, perm, count, list(bits), wkind, sub_k, sw_ref, True)
    assert np.array_equal(s_w.cpu().numpy().reshape(-1), np.asarray(sw_ref, np.float32).reshape(-1))
    ref = oracle.pack_act_rows(oracle.code_patterns(J, count, list(bits), wkind), count, list(bits), 128)
    assert np.array_equal(Wp.cpu().numpy(), ref)
