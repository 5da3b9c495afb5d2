"""Debug accumulators are [2][M][N] in every kernel: a layout with one group gives
zeros for the other."""
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


@pytest.mark.parametrize("M,flags", [(1, 0), (2, 0), (3, 0), (12, 1), (16, 0), (32, 0), (16, 16), (40, 2 | 4), (40, 2 | 8)])
@pytest.mark.parametrize("frac", [0.0, 1.0])
def test_absent_group_is_zero(sq, M, flags, frac):
    d = wl.random_linear(5, M, 300, 70, 4, 8, frac)
    lay = sq.Layout(d["perm"], d["count"], d["bits"])
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda())
    acc = torch.full((2, M, 70), -1, dtype=torch.int32, device="cuda")
    sq.mp_gemm(lay, Ap, s_a, Wp, s_w, acc_dbg=acc, flags=flags)
    assert sq.sync_status() == 0
    absent = int(frac == 0.0)
    assert not acc[absent].any() and acc[1 - absent].any()
