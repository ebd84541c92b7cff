"""The mode-3 DFT is a map of every tube by itself: tubes whose neighbours are
millions of times larger, or zero, are as accurate as they are alone.

Every tube (or lateral slice) is held to its own norm.  Tolerance: a length-n FFT
of a few passes errs by a small multiple of u log2(n), direct sums of length D by
about u sqrt(D); 8 u (log2 n + 1 + sqrt(n) / 4), and 8 times that for the worst
of many tubes.  The reference is numpy's transform in float64, one tube at a time (a
batched GPU transform of odd length may itself pair neighbouring tubes).
"""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# powers of two, products of small radices, even lengths with a direct part, odd products, odd with a direct part,
# primes, the longest
SIZES = [1, 2, 3, 4, 8, 9, 15, 17, 27, 32, 34, 45, 51, 64, 97, 100, 105, 128, 143, 187, 192, 225, 240, 255, 256, 257, 289, 331,
         334, 339, 384, 510, 512]
LONG = [720, 839, 993, 1000, 1001, 1022, 1024]


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


def rfft(x):
    return torch.from_numpy(np.fft.rfft(x.double().cpu().numpy(), axis=0)).cuda()


def tolerance(n, dtype):
    return 8 * 8 * torch.finfo(dtype).eps * (math.log2(n) + 1 + math.sqrt(n) / 4)


def norms(x):
    return x.abs().double().pow(2).sum(0).sqrt()


def check(tp, n, l, m, dtype, seed=0):
    g = torch.Generator(device="cuda").manual_seed(1000 * seed + n)
    scale = 10.0 ** torch.randint(-6, 7, (l, m), generator=g, device="cuda").double()
    scale[:, m // 2] = 0  # an all-zero lateral slice
    A = (torch.randn((n, l, m), generator=g, device="cuda", dtype=torch.float64) * scale).to(dtype)
    live = scale > 0
    ref = rfft(A)
    Ah = tp.fft(A)
    assert float((norms(Ah.to(ref.dtype) - ref) / norms(ref))[live].max()) < tolerance(n, dtype)
    assert float(Ah[:, ~live].abs().max()) == 0.0
    X = tp.ifft(ref.to(Ah.dtype).contiguous(), n)
    assert float((norms(X.double() - A.double()) / norms(A))[live].max()) < 2 * tolerance(n, dtype)
    assert float(X[:, ~live].abs().max()) == 0.0


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_every_tube_to_its_own_norm(tp, n, dtype):
    check(tp, n, 9, 8, dtype)
    check(tp, n, 5, 7, dtype)


@pytest.mark.parametrize("n", LONG)
def test_long_tubes_to_their_own_norm(tp, n):
    check(tp, n, 6, 7, torch.float32)


@pytest.mark.parametrize("n", [200, 240, 256, 143, 331, 334, 339, 510, 512])
@pytest.mark.parametrize("l,m", [(64, 38), (56, 44), (50, 50), (51, 49)])
def test_float64_on_both_sides_of_the_split(tp, n, l, m):
    """76 tiles of 32 tubes are split over more CTAs, 77 are not; a last tile that is full, in part, of odd count."""
    check(tp, n, l, m, torch.float64, seed=l)


@pytest.mark.parametrize("n", [48, 75, 97])
def test_unaligned_start_and_odd_slice_stride(tp, n):
    l, m = 5, 7
    buf = torch.randn(n * l * m + 1, device="cuda")
    A = buf[1:].view(n, l, m)
    ref = rfft(A)
    assert float((norms(tp.fft(A).to(ref.dtype) - ref) / norms(ref)).max()) < tolerance(n, torch.float32)


@pytest.mark.parametrize("n", [97, 225, 240, 256])
@pytest.mark.parametrize("factor", [1e-2, 1e-4, 1e-6])
def test_product_with_slices_of_different_scale(tp, n, factor):
    """Every lateral slice of A * B is as accurate as alone (the sizes take the Fourier form)."""
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, 40, 24), generator=g, device="cuda")
    B = torch.randn((n, 24, 2), generator=g, device="cuda")
    B[:, :, 1] *= factor
    C = tp.tprod(A, B).double()
    ref = torch.from_numpy(np.fft.irfft((rfft(A) @ rfft(B)).cpu().numpy(), n=n, axis=0)).cuda()
    # three transforms and sums of 24 products
    tol = 3 * tolerance(n, torch.float32) / 8 + 8 * torch.finfo(torch.float32).eps * math.sqrt(24)
    for j in range(2):
        assert float((C[:, :, j] - ref[:, :, j]).norm() / ref[:, :, j].norm()) < tol, j


@pytest.mark.parametrize("n", [15, 24, 31, 32])
def test_tgkb_slices_of_different_scale(tp, n):
    """tGKB_p solves every lateral slice as if it were alone: a dark frame beside a bright one, and an all-zero frame
    whose bound is zero.  The operator is well conditioned (3 times the t-identity and noise of norm about 1), so that a
    few steps meet the bounds and a solution errs by a few u times the condition number, 1e-5 at most."""
    N = 32
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, N, N), generator=g, device="cuda") * (0.5 / math.sqrt(n * N))
    A[0] += 3 * torch.eye(N, device="cuda")
    B = torch.randn((n, N, 3), generator=g, device="cuda")
    B[:, :, 1] *= 1e-6
    B[:, :, 2] = 0
    deltas = [1e-3 * float(B[:, :, j].norm()) for j in range(3)]
    X, infos = tp.tgkb_solve(A, B, max(deltas), 1.1, 20, deltas=deltas)
    for j in range(2):
        Y, info = tp.tgkb_solve(A, B[:, :, j:j + 1].contiguous(), deltas[j], 1.1, 20)
        assert infos[j]["status"] == 0 and infos[j]["k"] == info["k"]
        assert float((X[:, :, j] - Y[:, :, 0]).norm() / Y.norm()) < 1e-5
        R = tp.tprod(A, X[:, :, j:j + 1].contiguous()).double() - B[:, :, j:j + 1].double()
        assert float(R.norm()) < 1.1 * deltas[j] * (1 + 1e-3)
    assert infos[2]["status"] == 0 and float(X[:, :, 2].abs().max()) == 0.0
