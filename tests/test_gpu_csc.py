"""The CSC copy of a CSR input (csrc/k_csr.cu): column scan at block edges, the
bucket sort and its bitonic fallback (clustered rows), empty columns and rows.
A^T e_i products read single entries, so the transposed product is compared with
the FP64 one: each entry is one FMA chain over a column's c nonzeros, |error| <=
c 2^-24 sum |a x|."""
import numpy as np
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


def _csr(dense):
    m, n = dense.shape
    rows, cols = dense.nonzero()
    rowptr = np.zeros(m + 1, np.int64)
    np.add.at(rowptr, rows + 1, 1)
    return np.cumsum(rowptr).astype(np.int32), cols.astype(np.int32), dense[rows, cols]


def _pattern(kind, m, n, rng):
    D = np.zeros((m, n), np.float32)
    if kind == "uniform":
        D = (rng.random((m, n)) < 0.05) * rng.standard_normal((m, n))
    elif kind == "band":      # rows of a column lie close together
        i, j = np.indices((m, n))
        D = (np.abs(i - j * m // n) < 6) * rng.standard_normal((m, n))
    elif kind == "clustered":  # one far row, the rest in one bucket: bitonic
        D[:200, :] = rng.standard_normal((200, n))
        D[m - 1, :] = 1.0
    elif kind == "holes":     # empty columns and rows
        D[::7, ::5] = rng.standard_normal((len(range(0, m, 7)), len(range(0, n, 5))))
    return np.ascontiguousarray(D, dtype=np.float32)


@pytest.mark.parametrize("kind,m,n", [("uniform", 700, 1023), ("uniform", 1030, 1025),
                                      ("uniform", 300, 1), ("band", 3000, 500),
                                      ("clustered", 9000, 40), ("holes", 900, 2049)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_transposed_product(kind, m, n, dtype):
    rng = np.random.default_rng(m + n)
    rowptr, cols, vals = _csr(_pattern(kind, m, n, rng))
    v = torch.from_numpy(vals).cuda().to(dtype)
    A = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    r = torch.repeat_interleave(torch.arange(m), torch.from_numpy(np.diff(rowptr)).long()).cuda()
    A[r, torch.from_numpy(cols).long().cuda()] = v.double()
    X = torch.from_numpy(rng.standard_normal((m, 1)).astype(np.float32)).cuda()
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        args = (torch.from_numpy(rowptr).cuda(), torch.from_numpy(cols).cuda(), v, (m, n), X)
        Y = h.sketch_csr(*args, trans=True)
        assert torch.equal(Y, h.sketch_csr(*args, trans=True))
    finally:
        h.close()
    count = (A != 0).sum(0, dtype=torch.float64)[:, None]
    bound = (count + 1) * 2.0 ** -24 * (A.abs().T @ X.double().abs())
    assert bool(((Y.double() - A.T @ X.double()).abs() <= bound).all())
