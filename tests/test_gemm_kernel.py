"""Which kernel a few-row call runs: a FORCE flag means the kernel it names, and
without flags warp-level tensor instructions serve 3 <= M <= 32 where the rows fit."""
import ctypes

import pytest

from paper_2311_14114_gb300 import workloads as wl

GEMV, SKINNY = 1, 16
K_GEMV, K_FUSED, K_STAGED, K_SKINNY, K_ROWS = range(5)


@pytest.fixture(scope="module")
def sq():
    from paper_2311_14114_gb300 import build, soniq
    build.build()
    return soniq


def _kernel(sq, M, K, N, flags, bits=(4, 8), pad=128):
    c = sq.CLayout()
    c.K, c.n_groups, c.pad_unit = K, 2, pad
    c.count[0], c.count[1] = K - K // 4, K // 4
    for i in (0, 1):
        c.bits_w[i] = c.bits_a[i] = bits[i]
    return sq.lib().soniq_mp_gemm_kernel(ctypes.byref(c), M, N, flags, 0)


@pytest.mark.parametrize("M,K,flags,kernel", [
    (1, 512, 0, K_GEMV), (2, 512, 0, K_GEMV), (3, 512, 0, K_ROWS), (12, 512, 0, K_ROWS), (13, 512, 0, K_ROWS),
    (32, 512, 0, K_ROWS), (33, 512, 0, K_FUSED),
    (3, 512, GEMV, K_GEMV), (12, 512, GEMV, K_GEMV), (16, 512, GEMV, K_GEMV),
    (1, 512, SKINNY, K_SKINNY), (3, 512, SKINNY, K_SKINNY), (16, 512, SKINNY, K_SKINNY), (32, 512, SKINNY, K_SKINNY),
    (12, 7000, 0, K_GEMV), (12, 20000, 0, K_SKINNY), (16, 7000, 0, K_SKINNY)])
def test_kernel_of_few_rows(sq, M, K, flags, kernel):
    assert _kernel(sq, M, K, 300, flags) == kernel


def test_bad_arguments(sq):
    assert _kernel(sq, 0, 512, 300, 0) == -1
    assert _kernel(sq, 33, 512, 300, SKINNY) == -1


@pytest.mark.gpu
def test_rows_kernel_reports_a_lost_copy(sq):
    """The rows kernel's bounded wait, and that the context survives it."""
    torch = pytest.importorskip("torch")
    d = wl.random_linear(971, 16, 1000, 256, 3, 6, 0.25)
    lay = sq.Layout(d["perm"], d["count"], d["bits"])
    assert sq.gemm_kernel(lay, 16, 256) == sq.KERNEL_NAMES[K_ROWS]
    Wp, s_w = sq.pack_weights(lay, torch.from_numpy(d["W"]).cuda())
    Ap, s_a = sq.quantize_act(lay, torch.from_numpy(d["A"]).cuda())
    ref = sq.mp_gemm(lay, Ap, s_a, Wp, s_w, flags=SKINNY)
    assert sq.sync_status() == 0
    sq.mp_gemm(lay, Ap, s_a, Wp, s_w, flags=sq.FLAG_TEST_DROP_ARRIVE)
    assert sq.sync_status() == 5            # SONIQ_ERR_TIMEOUT, then cleared
    Y = sq.mp_gemm(lay, Ap, s_a, Wp, s_w)
    assert sq.sync_status() == 0
    assert torch.equal(Y.view(torch.int16), ref.view(torch.int16))
