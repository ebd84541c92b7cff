"""Small t-products, which are evaluated as the circular convolution itself,
against torch.fft in float64: every transpose, odd sizes, one to many columns,
sizes on both sides of the limit.

Tolerance: a sum of kk n products in float32 whose partial sums of kk terms are
added n at a time errs by at most about (kk + n) u relative to the sum of the
terms' magnitudes; random signs bring that to about sqrt(kk + n) u of the result's
scale.  8 u sqrt(kk + n).
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


@pytest.mark.parametrize("n,l,kk,m", [(1, 1, 1, 1), (1, 5, 3, 2), (2, 3, 1, 5), (3, 1, 7, 4), (8, 9, 5, 1), (16, 17, 31, 3),
                                      (31, 20, 10, 6), (32, 32, 32, 1), (33, 16, 8, 9), (64, 13, 12, 4), (100, 7, 11, 5),
                                      (127, 4, 9, 2), (128, 8, 8, 7), (129, 6, 6, 2), (24, 40, 40, 9), (32, 32, 32, 9)])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
def test_small_product(tp, n, l, kk, m, ta, tb):
    g = torch.Generator(device="cuda").manual_seed(n + l)
    A = torch.randn((n, kk, l) if ta else (n, l, kk), generator=g, device="cuda")
    B = torch.randn((n, m, kk) if tb else (n, kk, m), generator=g, device="cuda")
    C = tp.tprod(A, B, transA=ta, transB=tb)
    Ah, Bh = torch.fft.rfft(A.double(), dim=0), torch.fft.rfft(B.double(), dim=0)
    ref = torch.fft.irfft((Ah.mH if ta else Ah) @ (Bh.mH if tb else Bh), n=n, dim=0)
    u = torch.finfo(torch.float32).eps
    assert float((C.double() - ref).norm()) <= 8 * u * math.sqrt(kk + n) * float(ref.norm()) + 1e-30
