"""FP32 products whose operands come near the range limits of the three-part split
(csrc/k_f32tc.cu): which entries are formed again on the CUDA cores, alone and in
a batch, with the split skinny operand's image (no memory budget) and without."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[0, 1 << 35], ids=["image", "budget"])
def h(request):
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream, hbm_budget_bytes=request.param)
    yield h
    h.close()


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


@pytest.mark.parametrize("m,n,d", [(300, 260, 40), (70, 2600, 37), (1000, 520, 72)])
@pytest.mark.parametrize("trans", [False, True])
def test_zero_rows_stay_on_the_tensor_cores(h, m, n, d, trans):
    """A zero row (column) of A, or a zero column of X, beside one small element
    far from it: every other entry keeps the bits it has without that element."""
    g = _gen(m + n)
    A = torch.randn(m, n, generator=g, device="cuda")
    X = torch.randn(m if trans else n, d, generator=g, device="cuda")
    line = (lambda B, i: B[:, i]) if trans else (lambda B, i: B[i])
    line(A, 4).zero_()
    X[:, 3] = 0
    A[7, 9] = 0
    B = A.clone()
    B[7, 9] = 2.0 ** -60
    Y, Z = h.sketch(A, X, trans), h.sketch(B, X, trans)
    keep = torch.ones(Y.shape[0], dtype=torch.bool, device="cuda")
    keep[9 if trans else 7] = False
    assert torch.equal(Y[keep], Z[keep])
    assert bool((Z[4] == 0).all()) and bool((Z[:, 3] == 0).all())


@pytest.mark.parametrize("K", [127, 128, 300, 2600])
@pytest.mark.parametrize("trans", [False, True])
def test_products_that_underflow(h, K, trans):
    """Row 5 times column 2 is one product below the least normal number: FP32
    arithmetic holds it exactly."""
    g = _gen(K)
    M, d = 200, 20
    A = torch.randn(M, K, generator=g, device="cuda")
    X = torch.randn(K, d, generator=g, device="cuda")
    A[5] = 0
    A[5, 11] = 2.0 ** -75
    X[:, 2] = 0
    X[11, 2] = 3 * 2.0 ** -70
    Y = h.sketch(A.T.contiguous() if trans else A, X, trans)
    assert float(Y[5, 2]) == 3 * 2.0 ** -145
    R, S = A.double() @ X.double(), A.double().abs() @ X.double().abs()
    assert bool(((Y.double() - R).abs() <= (58 + K / 32) * 2.0 ** -24 * S + 2.0 ** -149).all())


@pytest.mark.parametrize("K", [127, 128, 2600])
@pytest.mark.parametrize("trans", [False, True])
def test_special_values(h, K, trans):
    g = _gen(K + 1)
    A = torch.randn(140, K, generator=g, device="cuda")
    X = torch.randn(K, 24, generator=g, device="cuda")
    for where in ("A", "X"):
        for bad in (float("inf"), float("-inf"), float("nan"), 2.0 ** 100, 2.0 ** -120):
            B, V = A.clone(), X.clone()
            (B if where == "A" else V)[9, 3] = bad
            Y = h.sketch(B.T.contiguous() if trans else B, V, trans)
            R, S = B.double() @ V.double(), B.double().abs() @ V.double().abs()
            F = R.float()
            assert torch.equal(torch.isnan(Y), torch.isnan(F))
            assert torch.equal(Y[torch.isinf(F)], F[torch.isinf(F)])
            ok = torch.isfinite(F)
            assert bool(((Y.double() - R).abs() <= (58 + K / 32) * 2.0 ** -24 * S)[ok].all())


@pytest.mark.parametrize("q", [0, 2])
def test_batch_items_equal_the_single_matrices(h, q):
    """Items inside the range, items formed again whole (an element below 2^-100)
    and items with zero rows, in one batch: each as alone, run after run."""
    g = _gen(q)
    As, Oms, ks = [], [], []
    for i, (m, n, k) in enumerate([(600, 300, 16), (500, 100, 24), (300, 900, 40), (257, 129, 9),
                                   (600, 300, 16), (2100, 1500, 64), (400, 700, 32)]):
        A = torch.randn(m, n, generator=g, device="cuda")
        if i in (1, 4, 5):
            A[3, 5] = 2.0 ** -110
        if i in (2, 3, 6):
            A[4] = 0
            A[:, 6] = 0
            A[7, 9] = 2.0 ** -60
        As.append(A)
        ks.append(k)
        Oms.append(torch.randn(n, k + 8, generator=g, device="cuda", dtype=torch.float64))
    want = [h.decompose(A, om, k, 8, q) for A, om, k in zip(As, Oms, ks)]
    b = h.prepare_batch(As, Oms, ks, 8, q)
    for _ in range(3):  # eager, captured, replayed
        for Q, L, P in b.outs:
            for t in (Q, L, P):
                t.fill_(float("nan"))
        b.run()
        for (Q, L, P), w in zip(b.outs, want):
            for x, y in zip((Q, L, P), w[:3]):
                assert torch.equal(x, y)


@pytest.mark.parametrize("m,n,d,i,j", [(20000, 1100, 96, 19999, 3), (20000, 1100, 96, 0, 1099),
                                       (700, 9000, 224, 300, 4500)])
@pytest.mark.parametrize("trans", [False, True])
def test_one_element_outside_the_range(h, m, n, d, i, j, trans):
    """The tensor-core product is given up in the middle: the whole result is the
    CUDA cores', and the next product runs as ever."""
    g = _gen(m + i)
    A = torch.randn(m, n, generator=g, device="cuda")
    X = torch.randn(m if trans else n, d, generator=g, device="cuda")
    want = h.sketch(A, X, trans)
    B = A.clone()
    B[i, j] = 2.0 ** 61
    Y = h.sketch(B, X, trans)
    Bt = B.double().T if trans else B.double()
    S = Bt.abs() @ X.double().abs()
    assert bool(((Y.double() - Bt @ X.double()).abs() <= X.shape[0] * 2.0 ** -24 * S).all())
    assert torch.equal(Y, h.sketch(B, X, trans))
    assert torch.equal(want, h.sketch(A, X, trans))


@pytest.mark.parametrize("m,K", [(300, 128), (300, 175), (300, 176), (39999, 175), (40000, 175)])
@pytest.mark.parametrize("d", [1, 7, 40])
@pytest.mark.parametrize("trans", [False, True])
def test_short_contractions_of_unaligned_rows(h, m, K, d, trans):
    """On both sides of the line between the CUDA cores and the tensor cores for
    operands whose rows are not on 16 bytes, with X a slice of a wider matrix."""
    g = _gen(m + K + d)
    A = torch.randn(K, m, generator=g, device="cuda") if trans else torch.randn(m, K, generator=g,
                                                                                device="cuda")
    X = torch.randn(K, d + 1, generator=g, device="cuda")[:, 1:]
    Y = h.sketch(A, X, trans)
    Ad = (A.T if trans else A).double()
    S = Ad.abs() @ X.double().abs()
    assert bool(((Y.double() - Ad @ X.double()).abs() <= (58 + K) * 2.0 ** -24 * S).all())
