"""t-products of shapes at the ends of what the entry points take: very many
columns or rows with little work, on both sides of the limits of the one-launch
form for small products, against torch.fft in float64.

Tolerance: sums of kk n float32 products of random signs err by about
u sqrt(kk + n) of the result's scale; 8 u sqrt(kk + n) + 8 u.
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


def reference(A, B):
    n = A.shape[0]
    return torch.fft.irfft(torch.fft.rfft(A.double(), dim=0) @ torch.fft.rfft(B.double(), dim=0), n=n, dim=0)


def tolerance(n, kk):
    return 8 * torch.finfo(torch.float32).eps * (math.sqrt(kk + n) + 1)


@pytest.mark.parametrize("n,l,kk,m", [(1, 1, 1, 262140), (1, 1, 1, 262141), (1, 1, 1, 300000), (2, 1, 4, 300000),
                                      (2, 1000000, 1, 1), (1, 1000000, 1, 3), (4, 3040, 2, 4), (4, 3041, 2, 4),
                                      (4, 760, 3, 16), (4, 760, 3, 17), (8, 3, 2, 7296), (8, 3, 2, 7297)])
def test_many_rows_or_columns(tp, n, l, kk, m):
    g = torch.Generator(device="cuda").manual_seed(l + m)
    A = torch.randn((n, l, kk), generator=g, device="cuda")
    B = torch.randn((n, kk, m), generator=g, device="cuda")
    C = tp.tprod(A, B).double()
    ref = reference(A, B)
    assert float((C - ref).norm() / ref.norm()) <= tolerance(n, kk)


@pytest.mark.parametrize("n,l,m", [(1, 4, 4), (8, 6, 5), (32, 32, 1), (33, 16, 9), (64, 12, 12), (240, 24, 6)])
@pytest.mark.parametrize("over", ["A", "B", "shifted"])
def test_result_over_an_operand(tp, n, l, m, over):
    """tprod_gemm with C at A, at B, or a slice past the start of B: small products and one of the Fourier form."""
    g = torch.Generator(device="cuda").manual_seed(n)
    if over == "A":
        m = l
    A = torch.randn((n, l, l), generator=g, device="cuda")
    buf = torch.randn((n + 1, l, m), generator=g, device="cuda")
    B = buf[:n]
    ref = reference(A, B)
    C = A if over == "A" else (B if over == "B" else buf[1:])
    L = tp.load()
    ws = torch.empty(L.tprod_gemm_workspace_bytes(l, l, m, n, 0) + 256, dtype=torch.uint8, device="cuda")
    wp = -(-ws.data_ptr() // 256) * 256
    st = L.tprod_gemm(A.data_ptr(), B.data_ptr(), C.data_ptr(), l, l, m, n, 0, 0, wp, ws.data_ptr() + ws.numel() - wp,
                      torch.cuda.current_stream().cuda_stream)
    assert st == 0
    assert float((C.double() - ref).norm() / ref.norm()) <= tolerance(n, l)
