"""RT-tSVD at the sizes up to which its blocks are taken: float64 blocks of one
and of four columns at 1024 rows and columns and at the largest ranks, and the
limit of wider blocks, max(l, m) + 2 r_max, on both sides."""
import numpy as np
import pytest
import torch

from oracle import methods as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


def problem(l, m, n, r, seed):
    """Singular values 1 .. 0.05 in r directions, 1e-4 noise in the data."""
    g = np.random.default_rng(seed)
    Ah = np.empty((n // 2 + 1, l, m), complex)
    for i in range(n // 2 + 1):
        real = i == 0 or 2 * i == n
        draw = lambda a: g.standard_normal((a, r)) + (0 if real else 1j) * g.standard_normal((a, r))
        U, V = np.linalg.qr(draw(l))[0], np.linalg.qr(draw(m))[0]
        Ah[i] = (U * np.geomspace(1, 0.05, r)) @ V.conj().T
    A = np.fft.irfft(Ah, n=n, axis=0)
    B = np.fft.irfft(Ah @ np.fft.rfft(g.standard_normal((n, m, 1)), axis=0), n=n, axis=0)
    E = g.standard_normal(B.shape)
    E *= 1e-4 * np.linalg.norm(B) / np.linalg.norm(E)
    return A, B + E, g.standard_normal((n, m, r)), float(np.linalg.norm(E))


def solve(tp, l, m, n, r, block, dtype=torch.float64):
    A, B, Om, delta = problem(l, m, n, r, l + r + block)
    dev = lambda a: torch.from_numpy(a).to("cuda", dtype)
    X, info = tp.rtsvd_solve(dev(A), dev(B), dev(Om), delta, 1.1, r - 1, block, 1, r_max=r, eps_rel=1e-12)
    ref = O.rtsvd_solve(A, B, Om, delta, 1.1, 1e-12 * np.sqrt(O.fro2(A)), r - 1, block, 1, r_max=r)
    assert info["r"] == ref["r"] == r
    if ref["margin"] > 1e-6:
        assert info["k"] == ref["k"]
        # backward stable at condition 20: far below 1e-10
        assert float(np.linalg.norm(X.cpu().numpy() - ref["X"]) / np.linalg.norm(ref["X"])) < 1e-10


@pytest.mark.parametrize("l,m,r,block", [(1024, 1024, 16, 1), (1024, 1024, 16, 4), (1024, 600, 18, 3), (780, 780, 16, 2),
                                         (300, 300, 256, 4), (1024, 300, 256, 4), (256, 1024, 256, 1)])
def test_float64_blocks_of_few_columns(tp, l, m, r, block):
    solve(tp, l, m, 2, r, block)


@pytest.mark.parametrize("block,limit", [(5, 811), (16, 811), (17, 308), (32, 308)])
def test_float64_limit_of_wider_blocks(tp, block, limit):
    r = 40
    solve(tp, limit - 2 * r, 64, 2, r, block)
    L = limit - 2 * r + 1
    z = lambda *s: torch.ones(s, device="cuda", dtype=torch.float64)
    with pytest.raises(tp.TprodError):
        tp.rtsvd_solve(z(2, L, 64), z(2, L, 1), z(2, 64, r), 1.0, 1.1, 4, block, 1, r_max=r, eps_rel=0.1)
