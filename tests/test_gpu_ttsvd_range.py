"""T-tSVD of operators whose range the leading columns do not span.

The slices have singular values 1 .. 0.1 in the columns that count (condition
10): errors of a backward stable solve are a modest multiple of u * 10 * sqrt(l);
40 u * 10 * sqrt(l) is the bound.
"""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


def wide(l, m, n, lead, seed):
    """(n, l, m) with m > l: a random core of condition 10, and leading columns of one kind."""
    rng = np.random.default_rng(seed)
    k = m - l
    Ah = np.zeros((n // 2 + 1, l, m), complex)
    for i in range(n // 2 + 1):
        real = i == 0 or 2 * i == n
        draw = lambda a, b: rng.standard_normal((a, b)) + (0 if real else 1j) * rng.standard_normal((a, b))
        U, V = np.linalg.qr(draw(l, l))[0], np.linalg.qr(draw(k, l))[0]
        Ah[i, :, l:] = (U * np.logspace(0, -1, l)) @ V.conj().T
        if lead == "repeated":
            Ah[i, :, :l] = Ah[i, :, l:l + 1]
        elif lead == "half":
            Ah[i, :, : l // 2] = draw(l, l // 2) / (3 * math.sqrt(l))
    return np.fft.irfft(Ah, n=n, axis=0), rng.standard_normal((n, l, 2))


@pytest.mark.parametrize("l,m,n", [(1, 3, 2), (5, 17, 3), (16, 40, 4), (24, 64, 5), (33, 70, 6), (100, 230, 2)])
@pytest.mark.parametrize("lead", ["zero", "repeated", "half"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_wide_operators(tp, l, m, n, lead, dtype):
    A, B = wide(l, m, n, lead, l + n)
    Ad, Bd = (torch.from_numpy(v).to("cuda", dtype) for v in (A, B))
    X, info, fac = tp.ttsvd_solve(Ad, Bd, 0.0, 1.1, keep=True)
    assert info["k"] == l and info["r"] == l
    Ah, Bh = (np.fft.rfft(v.double().cpu().numpy(), axis=0) for v in (Ad, Bd))
    ref = np.fft.irfft(np.linalg.pinv(Ah) @ Bh, n=n, axis=0)
    bound = 40 * torch.finfo(dtype).eps * 10 * math.sqrt(l)
    err = lambda x, r: np.linalg.norm(x.double().cpu().numpy() - r) / np.linalg.norm(r)
    assert err(X, ref) < bound
    # dL/dB = U S^{-1} V^T * G, the transposed solution operator
    G = np.random.default_rng(9).standard_normal((n, m, 2))
    Gd = torch.from_numpy(G).to("cuda", dtype)
    Gh = np.fft.rfft(Gd.double().cpu().numpy(), axis=0)
    dB = np.fft.irfft(np.linalg.pinv(Ah).conj().transpose(0, 2, 1) @ Gh, n=n, axis=0)
    assert err(tp.ttsvd_adjoint(fac, Gd), dB) < bound
