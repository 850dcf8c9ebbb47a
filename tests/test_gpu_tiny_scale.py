"""orth() of FP64 sketches so small that their Gram matrix is near or below the
least normal number (csrc/k_orth.cu): the same basis as at scale 1, which every
power of two leaves as it is.  Pass 1 sees a Gram of fewer bits; pass 2 restores
the basis to rounding level, so |Q - Q_1| <= 1e-10 kappa with kappa <= 100 here."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d", [(100, 5), (200, 30), (600, 300)])
@pytest.mark.parametrize("e", [-400, -510, -518, -520, -525])
def test_orth_fp64_of_tiny_sketches(M, d, e):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + d)
    Y = torch.randn(M, d, generator=g, device="cuda", dtype=torch.float64)
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        Q1 = h.orth(Y)
        Q = h.orth(Y * 2.0 ** e)
    finally:
        h.close()
    eye = torch.eye(d, device="cuda", dtype=torch.float64)
    assert float((Q.T @ Q - eye).abs().max()) <= 1e-13
    assert float((Q - Q1).abs().max()) <= 1e-8
