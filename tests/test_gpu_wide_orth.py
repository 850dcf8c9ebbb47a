"""orth() of FP32 sketches of 289 .. 512 columns (csrc/k_orth.cu): the factor in
shared memory up to 319 columns, in global memory above, where it is widened in
place.  CholeskyQR3 leaves |Q^T Q - I| at FP32 rounding (each entry a sum of M
products: 8 sqrt(M) 2^-24), and Q^T Y upper triangular with a positive diagonal to
the same relative level."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d", [(600, 289), (319, 319), (700, 320), (2000, 321), (513, 511),
                                 (512, 512), (20001, 400)])
def test_orth_fp32(M, d):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + d)
    # near-orthogonal columns of different sizes: a square Gaussian is ill conditioned
    Y = torch.eye(M, d, device="cuda") * 3 + torch.randn(M, d, generator=g, device="cuda") / M ** 0.5
    Y *= torch.logspace(0, 2, d, device="cuda")
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        Q = h.orth(Y)
    finally:
        h.close()
    u = 8 * M ** 0.5 * 2.0 ** -24
    Qd, Yd = Q.double(), Y.double()
    eye = torch.eye(d, device="cuda", dtype=torch.float64)
    assert float((Qd.T @ Qd - eye).abs().max()) <= u
    R = Qd.T @ Yd
    norms = Yd.norm(dim=0)
    assert float((R.tril(-1).abs() / norms).max()) <= u
    assert bool((R.diagonal() > 0).all())
    assert float(((Yd - Qd @ R).norm(dim=0) / norms).max()) <= u * d ** 0.5
