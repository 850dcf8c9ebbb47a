"""ruqlp_sketch into rows of a wider matrix: the result has the bits of the
contiguous call and nothing beside it is written, for rows on and off 16 bytes
(results go straight into the caller's rows where the kernels' stores allow), and
with Y over X (staged)."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    yield h
    h.close()


def _sketch(h, A, trans, X, d, Y, ldy):
    M = ruqlp.Matrix(0, ruqlp.Dense(A.shape[0], A.shape[1], A.stride(0),
                                    ruqlp._dtype_code(A.dtype), A.data_ptr()), ruqlp.Csr())
    h.check(ruqlp.ruqlp_sketch(h.h, M, int(trans), X.data_ptr(), X.stride(0), d, Y, ldy))


@pytest.mark.parametrize("dtype,m,n,d", [
    (torch.float64, 300, 200, 37), (torch.float64, 130, 700, 100), (torch.float32, 300, 90, 20),
    (torch.float32, 300, 1000, 37), (torch.float32, 1030, 640, 228), (torch.bfloat16, 300, 1000, 36),
    (torch.bfloat16, 4100, 1024, 220), (torch.bfloat16, 9000, 8200, 260),
    (torch.bfloat16, 500, 300, 7)])
@pytest.mark.parametrize("trans", [False, True])
def test_rows_of_a_wider_matrix(h, dtype, m, n, d, trans):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + d)
    n8 = (n + 7) // 8 * 8
    A = torch.randn(m, n8, generator=g, device="cuda", dtype=torch.float32).to(dtype)[:, :n]
    wt = torch.float64 if dtype == torch.float64 else torch.float32
    K, M = (m, n) if trans else (n, m)
    X = torch.randn(K, d, generator=g, device="cuda").to(wt)
    want = h.sketch(A, X, trans)
    for pad, off in ((0, 0), (1, 0), (4, 0), (4, 1), (12, 4)):
        buf = torch.full((M * (d + pad) + off + 8,), -7.0, dtype=wt, device="cuda")
        rows = buf[off:off + M * (d + pad)].view(M, d + pad)
        _sketch(h, A, trans, X, d, rows.data_ptr(), d + pad)
        assert torch.equal(rows[:, :d], want), (pad, off)
        assert bool((rows[:, d:] == -7).all()) and bool((buf[:off] == -7).all())
        assert bool((buf[off + M * (d + pad):] == -7).all())


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
def test_result_over_the_operand(h, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    A = torch.randn(512, 512, generator=g, device="cuda").to(dtype)
    wt = torch.float64 if dtype == torch.float64 else torch.float32
    X = torch.randn(512, 40, generator=g, device="cuda").to(wt)
    want = h.sketch(A, X)
    _sketch(h, A, False, X, 40, X.data_ptr(), 40)
    assert torch.equal(X, want)
