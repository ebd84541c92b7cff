"""The mode-3 DFT over tube lengths of every factorisation: products of small
radices (one to four passes), lengths with a part of larger primes (direct
sums), and the longest ones, on even and odd tube counts (paired and scalar
loads), against torch.fft in float64.

Tolerance: a length-n FFT of a few passes errs by a small multiple of
u log2(n); the direct sums of length D by about u sqrt(D) (random signs).
8 u (log2 n + sqrt(n) / 4) relative covers both with a margin.
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = list(range(1, 41)) + [49, 51, 64, 77, 96, 97, 100, 105, 121, 127, 143, 150, 169, 187, 192, 210, 225, 240, 255,
                              256, 257, 289, 320, 331, 339, 343, 360, 384, 391, 400, 405, 500, 509, 510, 512]
LONG = [513, 576, 600, 640, 720, 768, 810, 839, 899, 961, 1000, 1001, 1009, 1013, 1024]


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


def check(tp, n, l, m, dtype):
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, l, m), generator=g, device="cuda", dtype=dtype)
    u = torch.finfo(dtype).eps
    tol = 8 * u * (math.log2(n) + 1 + math.sqrt(n) / 4)
    ref = torch.fft.rfft(A.double(), dim=0)
    Ah = tp.fft(A)
    assert float((Ah.to(ref.dtype) - ref).norm() / ref.norm()) < tol
    X = tp.ifft(Ah, n)
    assert float((X.double() - A.double()).norm() / A.double().norm()) < 2 * tol
    # every tube by itself (no tube takes another's data)
    err = (Ah.to(ref.dtype) - ref).abs().pow(2).sum(0).sqrt() / ref.abs().pow(2).sum(0).sqrt()
    assert float(err.max()) < 8 * tol


@pytest.mark.parametrize("n", SIZES)
def test_every_factorisation(tp, n):
    check(tp, n, 9, 8, torch.float32)   # 72 tubes: two full tiles and a part
    check(tp, n, 5, 7, torch.float32)   # 35 tubes: scalar loads, an odd last tube
    check(tp, n, 3, 7, torch.float64)


@pytest.mark.parametrize("n", LONG)
def test_long_tubes(tp, n):
    check(tp, n, 6, 7, torch.float32)
    check(tp, n, 3, 11, torch.float32)


@pytest.mark.parametrize("n", [12, 17, 34, 256, 331])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_non_finite_tube_stays_alone(tp, n, value):
    A = torch.randn((n, 4, 8), device="cuda")
    ref = torch.fft.rfft(A.double(), dim=0)
    A[n // 2, 1, 3] = value
    Ah = tp.fft(A)
    bad = ~torch.isfinite(torch.view_as_real(Ah)).all(-1)
    assert bool(bad[:, 1, 3].all())
    bad[:, 1, 3] = False
    assert not bool(bad.any())
    ok = torch.ones(4, 8, dtype=torch.bool, device="cuda")
    ok[1, 3] = False
    assert float((Ah[:, ok].to(ref.dtype) - ref[:, ok]).norm() / ref.norm()) < 1e-5
    Xh = ref.to(torch.complex64).contiguous()
    Xh[1, 2, 5] = value
    X = tp.ifft(Xh, n)
    lost = ~torch.isfinite(X)
    assert bool(lost[:, 2, 5].any())
    lost[:, 2, 5] = False
    assert not bool(lost.any())


def test_unaligned_tensors_take_the_scalar_path(tp):
    """A tensor that starts 4 bytes past an 8-byte boundary, and an odd slice stride."""
    n, l, m = 48, 6, 8
    buf = torch.randn(n * l * m + 1, device="cuda")
    A = buf[1:].view(n, l, m)
    ref = torch.fft.rfft(A.double(), dim=0)
    Ah = tp.fft(A)
    assert float((Ah.to(ref.dtype) - ref).norm() / ref.norm()) < 1e-5
