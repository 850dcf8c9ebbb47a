"""Rounding error of FP64 products and Grams (csrc/k_simt.cu, k_fit), no larger
than that of chains of 16 products whose sums are added in turn (over K for a
product; over K slabs, then the slabs in turn, for a Gram).  Operands are FP32
values, so every product is exact in FP64 and the chains can be followed here;
the exact sums come from two-term compensated additions.  The errors are
compared in the root mean square over 2000 or more entries, whose sampling error
is below 3 %: at most 1.1 times."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


def _chains(P, slab):
    """Sums over dim 0 of P: chains of 16 in slabs of `slab` rows."""
    total = torch.zeros_like(P[0])
    for s0 in range(0, P.shape[0], slab):
        B = P[s0:s0 + slab]
        pad = -B.shape[0] % 16
        if pad:
            B = torch.cat([B, torch.zeros_like(B[:pad])])
        B = B.reshape(-1, 16, *B.shape[1:])
        part = torch.zeros_like(B[:, 0])
        for k in range(16):
            part = part + B[:, k]
        acc = torch.zeros_like(total)
        for b in range(part.shape[0]):
            acc = acc + part[b]
        total = total + acc
    return total


def _exact(P):
    hi = torch.zeros_like(P[0])
    lo = torch.zeros_like(hi)
    for k in range(P.shape[0]):
        x = P[k]
        s = hi + x
        t = s - hi
        lo = lo + ((hi - (s - t)) + (x - t))
        hi = s
    return hi, lo


def _rms(Y, exact):
    return float((((Y - exact[0]) - exact[1]) ** 2).mean().sqrt())


@pytest.fixture(scope="module")
def handle():
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    yield h
    h.close()


def _f32(g, *s):
    return torch.randn(*s, generator=g, device="cuda").double()


@pytest.mark.parametrize("K", [40, 64, 130, 300, 543, 544, 1000, 4096, 6000])
@pytest.mark.parametrize("M,N", [(70, 30), (40, 72)])
@pytest.mark.parametrize("trans", [False, True])
def test_product(handle, K, M, N, trans):
    g = torch.Generator(device="cuda")
    g.manual_seed(K + M)
    A = _f32(g, *((K, M) if trans else (M, K)))
    X = _f32(g, K, N)
    Y = handle.sketch(A, X, trans)
    Ak = A if trans else A.T.contiguous()
    P = Ak[:, :, None] * X[:, None, :]
    assert _rms(Y, _exact(P)) <= 1.1 * _rms(_chains(P, K), _exact(P))


@pytest.mark.parametrize("M,d", [(100, 64), (600, 50), (600, 100), (1000, 72), (2047, 64), (2048, 64),
                                 (8192, 50)])
def test_gram(handle, M, d):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + d)
    Y = _f32(g, M, d)
    G = handle.gram(Y)
    i, j = torch.triu_indices(d, d, 1, device="cuda")
    i, j = i[:4096], j[:4096]
    P = Y[:, i] * Y[:, j]
    tiles = (-(-d // 64)) ** 2
    splits = max(1, min((304 + tiles - 1) // tiles, -(-M // 64), 64))
    slab = -(--(-M // splits) // 16) * 16
    assert _rms(G[i, j], _exact(P)) <= 1.1 * _rms(_chains(P, slab), _exact(P))
    assert torch.equal(G, G.T)
