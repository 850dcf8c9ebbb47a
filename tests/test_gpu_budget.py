"""A handle's memory budget decides what is admitted, never a result: wide BF16
sketches of a matrix above 128 MB (one pass over A instead of two column
chunks) have the same bits, and need no more workspace, under the tightest
budget that admits them."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp
from paper_2209_12464_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _stream():
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("m,n,k", [(16384, 8192, 264), (8200, 8208, 250), (10000, 7000, 313),
                                   (8193, 8200, 376)])
def test_wide_bf16_is_the_same_under_a_budget(m, n, k):
    d = k + 8
    A = wl.aligned_rows(wl.dense_lowrank_gauss_torch(m + d, m, n, 40, noise_std=1e-3).bfloat16())
    Om = wl.omega_torch(d, n, d)
    need = ruqlp.ruqlp_workspace_bytes(m, n, d, ruqlp.BF16)
    free = ruqlp.Handle(0, _stream())
    tight = ruqlp.Handle(0, _stream(), hbm_budget_bytes=need)
    try:
        for trans in (False, True):
            X = Om.float() if not trans else wl.omega_torch(d + 1, m, d).float()
            assert torch.equal(free.sketch(A, X, trans), tight.sketch(A, X, trans))
        a, b = (h.decompose(A, Om, k, 8, 1) for h in (free, tight))
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x, y)
    finally:
        free.close()
        tight.close()


def test_served_wide_bf16_is_the_same_as_alone():
    m, n, k, p = 16384, 8192, 256, 16
    A = wl.aligned_rows(wl.dense_lowrank_gauss_torch(3, m, n, 40, noise_std=1e-3).bfloat16())
    Om = wl.omega_torch(4, n, k + p)
    torch.cuda.synchronize()
    server = ruqlp.Handle(0, _stream(), hbm_budget_bytes=8 << 30, max_slots=2)
    alone = ruqlp.Handle(0, _stream())
    try:
        ts = [server.submit(A, Om, k, p, 1, out_dtype=torch.float32) for _ in range(3)]
        while not all([server.poll(t) for t in ts]):
            pass
        ref = alone.decompose(A, Om, k, p, 1, out_dtype=torch.float32)
        for t in ts:
            for x, y in zip(t.outs, ref[:3]):
                assert torch.equal(x, y)
    finally:
        server.close()
        alone.close()
