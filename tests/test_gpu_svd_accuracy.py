"""Accuracy of the float32 small SVD: solutions of well-conditioned systems of
full rank by T-tSVD, against float64.

One-sided Jacobi whose rotations are applied with one rounded (c, s) to both
columns and to the right-hand sides (a kernel of eight lanes per pair of columns)
erred by BASE(r) u, the geometric mean over these eight systems of condition 3.
The present kernel may not be worse: a tenth is left for the order in which the
pairs come.
"""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BASE = {32: 8.84, 96: 18.18, 128: 22.56, 160: 27.90, 200: 32.08, 256: 46.18}


@pytest.fixture(scope="module")
def tp():
    from paper_2110_02485_gb300 import tprod
    tprod.load()
    return tprod


@pytest.mark.parametrize("r", sorted(BASE))
def test_error_of_a_full_rank_solution(tp, r):
    total = 0.0
    for s in range(8):
        rng = np.random.default_rng(1000 * r + s)
        Ah = []
        for _ in range(2):
            U = np.linalg.qr(rng.standard_normal((r, r)))[0]
            V = np.linalg.qr(rng.standard_normal((r, r)))[0]
            Ah.append((U * np.logspace(0, -math.log10(3.0), r)) @ V.T)
        A = np.stack([(Ah[0] + Ah[1]) / 2, (Ah[0] - Ah[1]) / 2])  # tubes of length 2: both spectral slices are real
        Ad = torch.from_numpy(A).to("cuda", torch.float32)
        Bd = torch.from_numpy(rng.standard_normal((2, r, 4))).to("cuda", torch.float32)
        X, info = tp.ttsvd_solve(Ad, Bd, 0.0, 1.1)
        assert info["k"] == r
        a, b = Ad.cpu().double().numpy(), Bd.cpu().double().numpy()
        x = [np.linalg.solve(a[0] + a[1], b[0] + b[1]), np.linalg.solve(a[0] - a[1], b[0] - b[1])]
        ref = np.stack([(x[0] + x[1]) / 2, (x[0] - x[1]) / 2])
        total += math.log(np.linalg.norm(X.cpu().double().numpy() - ref) / np.linalg.norm(ref))
    assert math.exp(total / 8) <= 1.1 * BASE[r] * torch.finfo(torch.float32).eps
