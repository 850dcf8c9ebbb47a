"""FP64 products, Grams and orthonormal bases at the edges of their fitted tiles
(k_fit in csrc/k_simt.cu, k_chol / k_trsm in csrc/k_orth.cu) against torch in
FP64.  Both sides round K products and sums: |difference| <= 2 (K + 72) 2^-53
sum |a x| (at most 8 + 64 slab sums besides)."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    handle = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    yield handle
    handle.close()


def _close(Y, A, X):
    bound = 2 * (X.shape[0] + 72) * 2.0 ** -53 * (A.abs() @ X.abs())
    assert bool(((Y - A @ X).abs() <= bound).all())


@pytest.mark.parametrize("m,n,d", [(1, 1, 1), (3, 130, 2), (65, 127, 3), (200, 513, 31),
                                   (1000, 800, 30), (777, 1001, 65), (2050, 300, 129),
                                   (600, 520, 512)])
@pytest.mark.parametrize("trans", [False, True])
def test_products(h, m, n, d, trans):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + d)
    A = torch.randn(m, n + 1, generator=g, device="cuda", dtype=torch.float64)[:, :n]
    X = torch.randn(m if trans else n, d, generator=g, device="cuda", dtype=torch.float64)
    _close(h.sketch(A, X, trans), A.T if trans else A, X)


@pytest.mark.parametrize("M,d", [(1, 1), (17, 5), (1000, 30), (500, 44), (333, 45), (4000, 89),
                                 (700, 512)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_gram(h, M, d, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + d)
    Y = torch.randn(M, d, generator=g, device="cuda", dtype=dtype)
    G = h.gram(Y)
    assert torch.equal(G, G.T)
    _close(G, Y.double().T, Y.double())


@pytest.mark.parametrize("M,d", [(1, 1), (40, 33), (1000, 30), (1216, 96), (2000, 97), (900, 512)])
def test_orth(h, M, d):
    """CholeskyQR2 of a well-conditioned Y: Q orthonormal and Y = Q R to a few
    d ulps (kappa(Y) below 100 keeps kappa^2 u far below both bounds)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + d)
    Y = torch.randn(M, d, generator=g, device="cuda", dtype=torch.float64)
    if M < 2 * d:  # a nearly square Gaussian is not: perturb an orthonormal basis
        Y = (torch.linalg.qr(Y)[0] + 1e-2 * Y / M ** 0.5).contiguous()
    Q = h.orth(Y)
    R = Q.T @ Y
    eye = torch.eye(d, device="cuda", dtype=torch.float64)
    assert (Q.T @ Q - eye).norm().item() <= 16 * d * 2.0 ** -52
    assert (torch.triu(R) - R).norm().item() <= 1e-12 * R.norm().item()
    assert bool((torch.diagonal(R) > 0).all())
    assert (Y - Q @ R).norm().item() <= 1e-13 * Y.norm().item()
