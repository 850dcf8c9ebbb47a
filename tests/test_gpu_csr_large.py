"""CSR with the largest number of nonzeros that int32 row pointers hold: every
loop over a row's entries ends at 2^31 - 1 (a 32-bit index plus a warp's stride
would not).  Ones times ones: the products are counts, exact in FP32."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


def test_csr_with_2_31_minus_1_nonzeros():
    m, n = 1024, 1 << 21
    nnz = m * n - 1
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    cols = torch.arange(n, dtype=torch.int32, device="cuda").repeat(m)[:nnz]
    rowptr = (torch.arange(m + 1, dtype=torch.int64, device="cuda") * n).clamp(max=nnz).int()
    vals = torch.ones(nnz, dtype=torch.bfloat16, device="cuda")
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        Y = h.sketch_csr(rowptr, cols, vals, (m, n), torch.ones(n, 4, device="cuda"))
        Z = h.sketch_csr(rowptr, cols, vals, (m, n), torch.ones(m, 4, device="cuda"), trans=True)
    finally:
        h.close()
    rows, columns = torch.full((m, 4), float(n)), torch.full((n, 4), float(m))
    rows[-1] -= 1
    columns[-1] -= 1
    assert torch.equal(Y.cpu(), rows)
    assert torch.equal(Z.cpu(), columns)
