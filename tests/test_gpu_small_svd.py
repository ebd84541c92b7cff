"""The small SVD (one-sided Jacobi) over ranks at the edges of its forms: one
block of four columns and parts of it, an odd number of blocks, the last and
first rank of every count of entries per lane, factors in shared memory and in
global memory, one and several right-hand sides.

T-tSVD at delta = 0 runs to full rank, so X is the solution of the slices'
linear systems and the residual history is fixed by the singular vectors.  The
slices have singular values 1 .. 0.1 (condition 10): errors of a backward
stable solve are a modest multiple of u * 10 * sqrt(r); 40 u * 10 * sqrt(r) is
the bound here.  The residuals are held to the same bound times ||B|| at every
k (the residual is Lipschitz in the leading subspace's projector only across
gaps, so the spectrum comes in well-separated groups and k at group ends).
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


def problem(r, m, n, p, seed):
    """A (n, r, m), its groups' ends, B; per-slice singular values in eight groups from 1 to 0.1."""
    rng = np.random.default_rng(seed)
    h = n // 2 + 1
    q = min(r, m)
    groups = min(8, q)
    ends = [q * (g + 1) // groups for g in range(groups)]
    s = np.concatenate([np.full(e - b, 10.0 ** (-g / max(1, groups - 1))) for g, (b, e) in enumerate(zip([0] + ends, ends))])
    s *= 1 + 0.02 * rng.random(q)
    Ah = np.empty((h, r, m), complex)
    for i in range(h):
        real = i == 0 or 2 * i == n
        draw = lambda a: rng.standard_normal((a, q)) + (0 if real else 1j) * rng.standard_normal((a, q))
        U, V = np.linalg.qr(draw(r))[0], np.linalg.qr(draw(m))[0]
        Ah[i] = (U * s) @ V.conj().T
    A = np.fft.irfft(Ah, n=n, axis=0)
    return A, rng.standard_normal((n, r, p)), ends


@pytest.mark.parametrize("r,p", [(1, 1), (2, 1), (3, 1), (4, 1), (5, 2), (8, 1), (9, 1), (12, 3), (13, 1), (31, 1), (32, 9),
                                 (33, 1), (64, 1), (65, 1), (96, 1), (97, 17), (128, 1), (129, 1), (160, 1), (160, 30),
                                 (161, 1), (168, 1), (169, 1), (192, 1), (193, 3), (224, 1), (225, 1), (256, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_full_rank_solution(tp, r, p, dtype):
    if dtype == torch.float64 and r > 130:
        pytest.skip("the float64 form does not change with the rank there")
    n = 3
    A, B, ends = problem(r, r, n, p, r)
    Ad, Bd = (torch.from_numpy(v).to("cuda", dtype) for v in (A, B))
    X, info, hist = tp.ttsvd_solve(Ad, Bd, 0.0, 1.1, res_hist=True)
    assert info["k"] == r and info["r"] == r
    bound = 40 * torch.finfo(dtype).eps * 10 * math.sqrt(r)
    Ah, Bh = (torch.fft.rfft(v.double(), dim=0) for v in (Ad, Bd))
    ref = torch.fft.irfft(torch.linalg.solve(Ah, Bh), n=n, dim=0)
    assert float((X.double() - ref).norm() / ref.norm()) < bound
    U = torch.linalg.svd(Ah)[0]
    beta = (U.mH @ Bh).abs().pow(2).sum(2)
    w = torch.tensor([1.0] + [2.0] * (n // 2), device="cuda", dtype=torch.float64)
    left = (w[:, None] * beta).flip(1).cumsum(1).flip(1).sum(0)  # sum over j >= k
    for k in ends[:-1]:
        want = math.sqrt(float(left[k]) / n)
        assert abs(hist[k] - want) < bound * float(Bd.double().norm()), k


@pytest.mark.parametrize("l,m", [(40, 24), (24, 40)])
def test_tall_and_wide(tp, l, m):
    n = 5
    A, B, _ = problem(l, m, n, 2, 3)
    Ad, Bd = (torch.from_numpy(v).to("cuda", torch.float32) for v in (A, B))
    X, info = tp.ttsvd_solve(Ad, Bd, 0.0, 1.1)
    Ah, Bh = (torch.fft.rfft(v.double(), dim=0) for v in (Ad, Bd))
    ref = torch.fft.irfft(torch.linalg.pinv(Ah) @ Bh, n=n, dim=0)
    assert float((X.double() - ref).norm() / ref.norm()) < 40 * 1.2e-7 * 10 * math.sqrt(24)


@pytest.mark.parametrize("l,m,n", [(64, 64, 331), (48, 40, 320), (16, 16, 609)])
def test_more_slices_than_multiprocessors(tp, l, m, n):
    """Two orthonormalisation blocks share a multiprocessor (row counts that are multiples of 16; 40 is not one)."""
    A, B, _ = problem(l, m, n, 1, 7)
    Ad, Bd = (torch.from_numpy(v).to("cuda", torch.float32) for v in (A, B))
    X, info = tp.ttsvd_solve(Ad, Bd, 0.0, 1.1)
    Ah, Bh = (torch.fft.rfft(v.double(), dim=0) for v in (Ad, Bd))
    ref = torch.fft.irfft(torch.linalg.pinv(Ah) @ Bh, n=n, dim=0)
    assert float((X.double() - ref).norm() / ref.norm()) < 40 * 1.2e-7 * 10 * math.sqrt(min(l, m))


def test_triplets_at_the_largest_working_set(tp):
    """tgkb_triplets with k = 119 fills the shared memory of the small SVD."""
    n, N, k = 2, 130, 119
    rng = np.random.default_rng(5)
    A = torch.from_numpy(rng.standard_normal((n, N, N))).to("cuda", torch.float32)
    B = torch.from_numpy(rng.standard_normal((n, N, 1))).to("cuda", torch.float32)
    U, S, V = tp.tgkb_triplets(A, B, k)
    Uh, Vh = (torch.fft.rfft(v.double(), dim=0) for v in (U, V))
    eye = torch.eye(k, device="cuda", dtype=torch.float64)
    assert float((Uh.mH @ Uh - eye).abs().max()) < 1e-3
    assert float((Vh.mH @ Vh - eye).abs().max()) < 1e-3
