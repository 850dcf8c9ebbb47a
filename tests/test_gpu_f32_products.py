"""FP32 products on the tensor cores (csrc/k_f32tc.cu) against FP64 products
of the same values, element by element.

Bound: the six part products are exact and the dropped ones below 2^-25 of
|a x|; a 32-deep block takes 12 truncating additions (2^-23 each) in the tensor
cores, the K / 32 block sums and the slab sums one rounding (2^-24) each, so
|error| <= (26 + K / 32 + slabs) 2^-24 sum |a x|, at most 32 slabs here."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handles():
    st = torch.cuda.current_stream().cuda_stream
    # a handle under a memory budget splits the skinny operand in every CTA
    hs = ruqlp.Handle(0, st), ruqlp.Handle(0, st, hbm_budget_bytes=1 << 35)
    yield hs
    for h in hs:
        h.close()


def _ref(A, X, trans):
    A, X = A.double(), X.double()
    A = A.T if trans else A
    return A @ X, A.abs() @ X.abs()


def _check(Y, A, X, trans):
    R, S = _ref(A, X, trans)
    bound = (58 + X.shape[0] / 32) * 2.0 ** -24 * S
    assert bool(((Y.double() - R).abs() <= bound).all())


@pytest.mark.parametrize("m,n,d", [(64, 200, 1), (128, 128, 16), (257, 255, 17), (300, 1000, 33),
                                   (1001, 777, 37), (2560, 2047, 224), (640, 20000, 225),
                                   (512, 300, 300), (19500, 1030, 20)])
@pytest.mark.parametrize("trans", [False, True])
def test_products(handles, m, n, d, trans):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + d)
    for pad in (0, 1, 4):  # rows on and off 16-byte boundaries
        A = torch.randn(m, n + pad, generator=g, device="cuda")[:, :n]
        X = torch.randn(m if trans else n, d + pad, generator=g, device="cuda")[:, :d]
        Y = handles[0].sketch(A, X, trans)
        _check(Y, A, X, trans)
        assert torch.equal(Y, handles[1].sketch(A, X, trans))


@pytest.mark.parametrize("trans", [False, True])
def test_special_values_and_range(handles, trans):
    """Infinities and NaN reach the outputs they reach in FP32; magnitudes near
    FP32's limits, and rows far below the rest, keep FP32 accuracy."""
    h = handles[0]
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.randn(300, 260, generator=g, device="cuda")
    X = torch.randn(300 if trans else 260, 40, generator=g, device="cuda")
    r = (lambda B, i: B[:, i]) if trans else (lambda B, i: B[i])
    for bad in (float("inf"), float("-inf"), float("nan")):
        B = A.clone()
        B[7, 7] = bad
        Y, R = h.sketch(B, X, trans), _ref(B, X, trans)[0].float()
        assert torch.equal(torch.isnan(Y), torch.isnan(R))
        assert torch.equal(torch.isinf(Y), torch.isinf(R))
        assert torch.equal(Y[torch.isinf(R)], R[torch.isinf(R)])
    for a, x in ((1e30, 1e6), (1e-20, 1e-15), (2.0 ** -126, 1e6), (1.0, 1e-30)):
        _check(h.sketch(A * a, X * x, trans), A * a, X * x, trans)
    B = A.clone()
    r(B, 3).mul_(1e-33)
    r(B, 4).zero_()
    Y = h.sketch(B, X, trans)
    _check(Y, B, X, trans)
    assert bool((Y[4] == 0).all())


@pytest.mark.parametrize("m,n,d", [(4100, 1024, 220), (2049, 520, 16), (5000, 4096, 224),
                                   (16392, 4104, 257), (4100, 16400, 272), (8200, 8207, 384),
                                   (640, 808, 272), (500, 1200, 385), (20000, 4096, 220)])
@pytest.mark.parametrize("trans", [False, True])
def test_bf16_products_pairs_and_wide(handles, m, n, d, trans):
    """BF16 products with the tuner free (CTA pairs among its choices) and of more
    than 256 columns in one pass.  Every addition of a K-long accumulation may be
    truncated by the tensor core: |error| <= (K / 16 + 160) 2^-23 sum |a x|."""
    h = handles[0]
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + d)
    n8 = (n + 7) // 8 * 8
    A = torch.randn(m, n8, generator=g, device="cuda").bfloat16()[:, :n]
    X = torch.randn(m if trans else n, d, generator=g, device="cuda")
    Y = h.sketch(A, X, trans)
    R, S = _ref(A, X.bfloat16(), trans)
    assert bool(((Y.double() - R).abs() <= (X.shape[0] / 16 + 160) * 2.0 ** -23 * S).all())
    assert torch.equal(Y, h.sketch(A, X, trans))
    # a handle under a budget takes wide sketches in column chunks
    Z = handles[1].sketch(A, X, trans)
    assert bool(((Z.double() - R).abs() <= (X.shape[0] / 16 + 160) * 2.0 ** -23 * S).all())
