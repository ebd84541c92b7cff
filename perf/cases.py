"""The calls that programs built on this framework make, as timed cases.

The listed cases follow the workloads of the package's own configurations
(`synth.CONFIGS`, the uneven batch, the video batch, the differentiation
form): the bare t-product and transform, the five solvers, the batched forms
and the gradients.  Each goes through the public functions of `tprod` on
tensors that a program has on the GPU before the call.

`draw` gives more calls of the same kinds over the whole range of sizes:
square and rectangular slices, odd and non-power-of-two tube lengths, one to 32
lateral slices, float32, float64 and the two reduced forms of the sketch.

`exact` restates each call in float64 with plain torch and numpy.
"""
from __future__ import annotations

import concurrent.futures
import math

import numpy as np
import torch

from paper_2110_02485_gb300 import synth, tprod

DEVICE = "cuda"


def listed() -> list:
    return [
        # a single small product: one image row blurred by a 32^3 operator; launches and latency only
        dict(name="product_32", op="product", l=32, kk=32, m=1, n=32, dtype="float32"),
        # the forward blur of six RGB-like planes of a 240 x 240 image (a tube length that is no power of two)
        dict(name="product_240_p6", op="product", l=240, kk=240, m=6, n=240, dtype="float32"),
        # learning an operator: the t-product of 32 frames and both its gradients
        dict(name="product_grad_256_p32", op="product_grad", l=256, kk=256, m=32, n=256, dtype="float32"),
        # transforming an operator once for several solves, and back (the largest size of the uneven batch)
        dict(name="spectrum_384", op="spectrum", l=384, m=384, n=384, dtype="float32"),
        # the plain float64 method on one 32^3 problem: T-tSVD, RT-tSVD and tGKB
        dict(name="plain_32_float64", op="plain", N=32, n=32, sigma=1.5, band=4, s=2.0, noise=1e-2, tau=1.01,
             p_over=5, block=1, r_max=32, eps_rel=3e-2, k_max=32, dtype="float64"),
        # image deblurring, the size the throughput figure is quoted on
        dict(name="rtsvd_256", op="rtsvd", N=256, n=256, p=1, sigma=2.5, band=8, s=3.0, noise=1e-3, tau=1.1,
             p_over=10, block=16, r_max=160, eps_rel=2e-2, form="fp32"),
        # the precision form at 512^3: the sketch's products in tf32
        dict(name="rtsvd_512_tf32", op="rtsvd", N=512, n=512, p=1, sigma=3.0, band=12, s=4.0, noise=1e-3, tau=1.1,
             p_over=10, block=16, r_max=160, eps_rel=10 ** -1.2, form="tf32"),
        # the same image by Tikhonov-tGKB (tGKB and the search of the parameter)
        dict(name="tgkt_256", op="tgkt", N=256, n=256, sigma=2.5, band=8, s=3.0, noise=1e-3, tau=1.1, k_max=100),
        # video: 32 frames as lateral slices, each with its own bound (tGKB_p)
        dict(name="video_tgkb_256_p32", op="tgkb", N=256, n=256, p=32, sigma=2.5, band=8, s=3.0, noise=1e-3, tau=1.2,
             k_max=100),
        # independent problems of uneven sizes, RT-tSVD and tGKB each, replayed as one CUDA graph over four streams
        dict(name="uneven_batch", op="batch", sizes="64,96,128,192,256,320,384", noise=1e-2, tau=1.1, eps_j=6),
        # learning the blur: the tGKB solution and its gradients in the data and the tube weights
        dict(name="tgkb_grad_256", op="grad", method="tgkb", N=256, n=256, sigma=2.5, band=8, s=3.0, noise=1e-2,
             tau=1.1, k_max=100),
        # the full T-tSVD of the image problem, which the paper compares RT-tSVD with
        dict(name="ttsvd_256", op="ttsvd", N=256, n=256, sigma=2.5, band=8, s=3.0, noise=1e-3, tau=1.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    op = rng.choice(("product", "product", "product_grad", "spectrum", "rtsvd", "rtsvd", "tgkt", "tgkb", "ttsvd",
                     "batch", "grad", "plain"))
    if op in ("product", "product_grad", "spectrum"):
        double = rng.random() < 0.2
        top = 96 if double else 384
        l, kk, n = (_log_int(rng, 24, top) for _ in range(3))
        dtype = "float64" if double else "float32"
        if op == "spectrum":
            return dict(op=op, l=l, m=kk, n=n, dtype=dtype)
        return dict(op=op, l=l, kk=kk, m=_log_int(rng, 1, 96), n=n, dtype=dtype)
    blur = dict(sigma=rng.uniform(1.5, 3.0), band=rng.randint(4, 12), s=rng.uniform(2.0, 4.0))
    noise = math.exp(rng.uniform(math.log(3e-3), math.log(2e-2)))
    if op == "plain":
        N = _log_int(rng, 16, 40)
        return dict(op=op, N=N, n=_log_int(rng, 16, 40), sigma=1.5, band=4, s=2.0, noise=1e-2, tau=1.01, p_over=5,
                    block=rng.randint(1, 5), r_max=N, eps_rel=3e-2, k_max=N, dtype="float64")
    if op == "batch":
        return dict(op=op, sizes=",".join(str(_log_int(rng, 48, 300)) for _ in range(rng.randint(2, 5))),
                    noise=noise, tau=1.1, eps_j=rng.randint(5, 7))
    N, n = _log_int(rng, 40, 320), _log_int(rng, 40, 400)
    if op == "ttsvd":
        # a cut inside a cluster of singular values is ill-posed in float32: the image problem's blur and noise
        return dict(op=op, N=_log_int(rng, 128, 256), n=_log_int(rng, 32, 160), noise=noise / 10, tau=1.1, sigma=2.5,
                    band=8, s=3.0)
    if op == "tgkt":
        return dict(op=op, N=N, n=n, noise=noise, tau=1.1, k_max=min(N, 100), **blur)
    if op == "tgkb":
        return dict(op=op, N=N & ~1, n=n, p=_log_int(rng, 1, 24), noise=noise, tau=1.2, k_max=min(N & ~1, 60), **blur)
    if op == "grad":
        return dict(op=op, method=rng.choice(("tgkb", "rtsvd")), N=N, n=n, noise=noise, tau=1.1, k_max=min(N, 100),
                    p_over=10, block=16, r_max=min(N, 128), eps_rel=0.2, **blur)
    form = rng.choice(("fp32", "fp32", "tf32", "bf16"))
    if form == "bf16":  # rows of 16 bytes
        N = min(N, 128) & ~3
    return dict(op=op, N=N, n=n, p=_log_int(rng, 1, 8), noise=noise, tau=1.1, p_over=10,
                block=rng.choice((8, 16, 16)), r_max=min(N, 160), eps_rel=0.2, form=form, **blur)


# ---- inputs ---------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _operator(N, n, sigma, band, s):
    T, c = synth.blur_factors(N, sigma, band, s, n)
    return torch.from_numpy(T).to(DEVICE), torch.from_numpy(c).to(DEVICE)


def _data(N, n, p, sigma, band, s, noise, rng):
    """p blurred noisy images (or frames of one scene) as lateral slices, and each slice's bound."""
    T, c = synth.blur_factors(N, sigma, band, s, n)
    bumps, rects = (5, 2) if N <= 40 else (20, 4)
    imgs = synth.synthetic_video(N, n, p, bumps, rects, rng) if p > 1 else \
        synth.synthetic_image(N, n, bumps, rects, rng)[None]
    circ = c[(np.arange(n)[:, None] - np.arange(n)[None, :]) % n]
    clean = np.matmul(np.matmul(T, imgs), circ.T)
    B, _ = synth.add_noise(clean, noise, rng)
    lateral = lambda v: torch.from_numpy(np.ascontiguousarray(v.transpose(2, 1, 0)).astype(np.float32)).to(DEVICE)
    return lateral(B), [float(np.linalg.norm(e)) for e in B - clean]


def _problem(case, seed, N, n, p=1, r_max=0, **over):
    """One deblurring problem on the GPU (A, B, Omega, the blur's factors, the bounds)."""
    q = dict(sigma=2.5, band=8, s=3.0, noise=1e-2)
    q.update({k: case[k] for k in q if k in case})
    q.update(over)
    T, c = _operator(N, n, q["sigma"], q["band"], q["s"])
    B, deltas = _data(N, n, p, q["sigma"], q["band"], q["s"], q["noise"], synth.rng_for(seed))
    d = dict(A=(c[:, None, None] * T).float(), B=B, T=T.float(), c=c.float(), deltas=deltas,
             delta=float(np.linalg.norm(deltas)))
    if r_max:
        d["Omega"] = torch.randn((n, N, r_max), generator=_generator(seed), device=DEVICE)
    return d


def _problems(case, seed):
    """The problems of an uneven batch with the solver arguments that its sizes ask for."""
    out = []
    for i, N in enumerate(int(v) for v in case["sizes"].split(",")):
        d = _problem(case, seed + 101 * i, N, N, r_max=min(N, synth.UNEVEN_R_CAP))
        d.update(eps_rel=10.0 ** (-case["eps_j"] / 10.0), k_max=min(N, synth.UNEVEN_KMAX))
        out.append(d)
    return out


def _solve_batch(problems, side, tau):
    """Every problem's two solves, over the side streams, joined at the end."""
    main = torch.cuda.current_stream()
    out = [None] * len(problems)
    for st in side:
        st.wait_stream(main)
    for i, d in enumerate(problems):
        with torch.cuda.stream(side[i % len(side)]):
            X, info, _ = tprod.rtsvd_solve(d["A"], d["B"], d["Omega"], d["delta"], tau, synth.UNEVEN_P_OVER,
                                           synth.UNEVEN_BLOCK, synth.UNEVEN_Q, d["Omega"].shape[2],
                                           eps_rel=d["eps_rel"], sync=False)
            Y, jnfo, _ = tprod.tgkb_solve(d["A"], d["B"], d["delta"], tau, d["k_max"], sync=False)
            out[i] = (X, Y, info, jnfo)
    for st in side:
        main.wait_stream(st)
    return out


def _cotangent(case, seed):
    """dL/dX of a smooth loss: image-like, one lateral slice."""
    img = synth.synthetic_image(case["N"], case["n"], 20, 4, synth.rng_for(seed + 1))
    return torch.from_numpy(synth.lateral(img).astype(np.float32)).to(DEVICE)


def prepare(case, seed):
    op = case["op"]
    if op in ("product", "product_grad"):
        dtype = getattr(torch, case["dtype"])
        g = _generator(seed)
        l, kk, m, n = case["l"], case["kk"], case["m"], case["n"]
        st = dict(case=case, A=torch.randn((n, l, kk), generator=g, device=DEVICE, dtype=dtype),
                  B=torch.rand((n, kk, m), generator=g, device=DEVICE, dtype=dtype))
        if op == "product_grad":
            st["A"].requires_grad_()
            st["B"].requires_grad_()
            st["G"] = torch.randn((n, l, m), generator=g, device=DEVICE, dtype=dtype)
        return st
    if op == "spectrum":
        A = torch.randn((case["n"], case["l"], case["m"]), generator=_generator(seed), device=DEVICE,
                        dtype=getattr(torch, case["dtype"]))
        return dict(case=case, A=A)
    if op == "batch":
        problems = _problems(case, seed)
        side = [torch.cuda.Stream() for _ in range(4)]
        # the graph holds the solves' workspaces; its inputs stay in `problems`
        graph = tprod.Captured(lambda: _solve_batch(problems, side, case["tau"]), warmup=1)
        return dict(case=case, problems=problems, graph=graph)
    d = _problem(case, seed, case["N"], case["n"], case.get("p", 1), case.get("r_max", 0))
    d["case"] = case
    if op == "plain":
        for k in ("A", "B", "Omega"):
            d[k] = d[k].double()
    if op == "grad":
        d["c"].requires_grad_()
        d["B"].requires_grad_()
        d["G"] = _cotangent(case, seed)
    return d


MU_LO, MU_HI = synth.CONFIGS["n256"].mu_lo, synth.CONFIGS["n256"].mu_hi


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "product":
        return tprod.tprod(st["A"], st["B"])
    if op == "product_grad":
        C = tprod.tprod_ad(st["A"], st["B"])
        dA, dB = torch.autograd.grad(C, (st["A"], st["B"]), st["G"])
        return dict(C=C, dA=dA, dB=dB)
    if op == "spectrum":
        Ah = tprod.fft(st["A"])
        return dict(spectrum=Ah, back=tprod.ifft(Ah, case["n"]))
    if op == "batch":
        return [dict(rtsvd=X, tgkb=Y) for X, Y, _, _ in st["graph"].replay()]
    A, B, delta, tau = st["A"], st["B"], st["delta"], case["tau"]
    if op == "rtsvd":
        X, info = tprod.rtsvd_solve(A, B, st["Omega"], delta, tau, case["p_over"], case["block"], 1, case["r_max"],
                                    eps_rel=case["eps_rel"], tf32=case["form"] == "tf32", bf16=case["form"] == "bf16")
        return dict(X=X, k=info["k"], r=info["r"])
    if op == "tgkt":
        X, info = tprod.tgkt_solve(A, B, delta, tau, case["k_max"], MU_LO, MU_HI)
        return dict(X=X, k=info["k"])
    if op == "tgkb":
        X, infos = tprod.tgkb_solve(A, B, delta, tau, case["k_max"],
                                    deltas=st["deltas"] if case["p"] > 1 else None)
        return dict(X=X, k=[i["k"] for i in (infos if case["p"] > 1 else [infos])])
    if op == "ttsvd":
        X, info = tprod.ttsvd_solve(A, B, delta, tau)
        return dict(X=X, k=info["k"])
    if op == "plain":
        T, ti = tprod.ttsvd_solve(A, B, delta, tau)
        R, ri = tprod.rtsvd_solve(A, B, st["Omega"], delta, tau, case["p_over"], case["block"], 1, case["r_max"],
                                  eps_rel=case["eps_rel"])
        G, gi = tprod.tgkb_solve(A, B, delta, tau, case["k_max"])
        return dict(ttsvd=T, rtsvd=R, tgkb=G, k=[ti["k"], ri["k"], gi["k"]])
    # grad: what the layers after the solve hand back (G) taken to the data and the tube weights, at the solve's k
    if case["method"] == "tgkb":
        X = tprod.tgkb_solve_ad(A, B, delta, tau, case["k_max"])
        (dB,) = torch.autograd.grad(X, (B,), st["G"])
        dc = tprod.sep_grad_c(X.detach(), st["G"], st["c"].detach().double()).float()
    else:
        X = tprod.rtsvd_solve_sep_ad(st["c"].double(), st["T"], B, st["Omega"], delta, tau, case["p_over"],
                                     block=case["block"], q_power=1, r_max=case["r_max"], eps_rel=case["eps_rel"])
        dB, dc = torch.autograd.grad(X, (B, st["c"]), st["G"])
    return dict(X=X, dB=dB, dc=dc)


# ---- the work that no implementation can do without ------------------------------

def _fft_flops(n, tubes):
    return 2.5 * n * math.log2(max(n, 2)) * tubes


def _rt_flops(N, n, r, p=1, q=1):
    h = n // 2 + 1
    products = 8.0 * h * N * N * r * (2 + 2 * q + 1)  # sketch, power passes, projection, K = A V
    orth = 8.0 * h * N * r * r * (2 + q)              # orthonormalisation of the sketch, the passes and B^H
    svd = 8.0 * h * 10.0 * r ** 3
    return products + orth + svd + _fft_flops(n, N * (N + r + 2 * p))


def _gk_flops(N, n, k, p=1):
    h = n // 2 + 1
    return p * h * (16.0 * N * N * k + 32.0 * N * k * k) + _fft_flops(n, N * (N + 2 * p))


def work(case):
    op, n = case["op"], case.get("n", 0)
    if op in ("product", "product_grad"):
        e = 8 if case["dtype"] == "float64" else 4
        l, kk, m = case["l"], case["kk"], case["m"]
        times = 1 if op == "product" else 3
        size = n * (l * kk + kk * m + l * m) * e
        return dict(bytes=size if op == "product" else 2 * size,
                    flops=times * (8.0 * (n // 2 + 1) * l * kk * m) + _fft_flops(n, (l * kk + kk * m + l * m)) * (
                        1 if op == "product" else 2))
    if op == "spectrum":
        e = 8 if case["dtype"] == "float64" else 4
        tubes = case["l"] * case["m"]
        return dict(bytes=2 * tubes * e * (n + 2 * (n // 2 + 1)), flops=2 * _fft_flops(n, tubes))
    if op == "batch":
        w = dict(bytes=0, flops=0.0)
        for N in (int(v) for v in case["sizes"].split(",")):
            r = min(N, synth.UNEVEN_R_CAP)
            w["bytes"] += 4 * (N ** 3 + N * N * r + 3 * N * N)
            w["flops"] += _rt_flops(N, N, r / 2) + _gk_flops(N, N, 8)
        return w
    N, p = case["N"], case.get("p", 1)
    e = 8 if op == "plain" else 4
    size = e * (n * N * N + 2 * n * N * p)
    if op in ("rtsvd", "plain") or case.get("method") == "rtsvd":
        size += e * n * N * case["r_max"]
    if op == "rtsvd":
        flops = _rt_flops(N, n, 0.6 * case["r_max"], p)
    elif op == "ttsvd":
        flops = 8.0 * (n // 2 + 1) * 20.0 * N ** 3
    elif op == "plain":
        flops = 8.0 * (n // 2 + 1) * 20.0 * N ** 3 + _rt_flops(N, n, N / 2) + _gk_flops(N, n, 8)
    elif op == "grad":
        flops = 2 * _rt_flops(N, n, 0.5 * case["r_max"]) if case["method"] == "rtsvd" else 3 * _gk_flops(N, n, 8)
    else:
        flops = _gk_flops(N, n, 20, p)
    return dict(bytes=size, flops=flops)


# ---- the same calls in float64 ----------------------------------------------------

def _weights(n):
    h = n // 2 + 1
    w = torch.full((h,), 2.0, dtype=torch.float64, device=DEVICE)
    w[0] = 1.0
    if n % 2 == 0:
        w[-1] = 1.0
    return w


def _hat(x):
    return torch.fft.rfft(x.double(), dim=0)


def _svd(M):
    """Singular value decompositions of a stack of matrices, on the host (LAPACK, a thread per part)."""
    M = M.cpu().numpy()
    parts = np.array_split(np.arange(M.shape[0]), min(16, M.shape[0]))
    with concurrent.futures.ThreadPoolExecutor(16) as ex:
        got = list(ex.map(lambda i: np.linalg.svd(M[i], full_matrices=False), parts))
    return tuple(torch.from_numpy(np.concatenate([g[j] for g in got])).to(DEVICE) for j in range(3))


def _orth(Y, Q=None):
    if Q is not None and Q.shape[2]:
        for _ in range(2):
            Y = Y - Q @ (Q.mH @ Y)
    return torch.linalg.qr(Y)[0]


def _truncated(V, S, beta, Ah, Bh, n, k_init, r, bound):
    """The discrepancy principle over k in [k_init, r] for X = V_k S_k^-1 beta_k."""
    w = _weights(n)
    alpha = beta / S[:, :, None]
    K = Ah @ V
    R = Bh - K[:, :, :k_init - 1] @ alpha[:, :k_init - 1]
    k = r
    for j in range(k_init, r + 1):
        R = R - K[:, :, j - 1:j] @ alpha[:, j - 1:j]
        res = math.sqrt(float((w[:, None, None] * R.abs() ** 2).sum()) / n)
        if res <= bound:
            k = j
            break
    return k, V[:, :, :k] @ alpha[:, :k]


def _exact_rtsvd(d, tau, p_over, block, r_max, eps_rel, full=False):
    """RT-tSVD by its definition (block sketch, one power iteration, SVD of the projection, discrepancy principle)."""
    n = d["A"].shape[0]
    Ah, Bh, Oh = _hat(d["A"]), _hat(d["B"]), _hat(d["Omega"])
    w = _weights(n)
    eta = float((d["A"].double() ** 2).sum())
    eps2 = eps_rel * eps_rel * eta
    Q = Ah.new_zeros((Ah.shape[0], Ah.shape[1], 0))
    BH = Ah.new_zeros((Ah.shape[0], Ah.shape[2], 0))
    r = 0
    while eta >= eps2 and r < r_max:
        bb = min(block, r_max - r)
        Y = _orth(Ah @ Oh[:, :, r:r + bb], Q)
        Y = _orth(Ah @ _orth(Ah.mH @ Y), Q)
        Z = Ah.mH @ Y
        eta -= float((w[:, None, None] * Z.abs() ** 2).sum()) / n
        Q, BH, r = torch.cat([Q, Y], 2), torch.cat([BH, Z], 2), r + bb
    QG, R = torch.linalg.qr(BH)
    UR, S, UbH = _svd(R)  # BH = (QG UR) S Ub^H
    V = QG @ UR
    k, Xh = _truncated(V, S, UbH @ (Q.mH @ Bh), Ah, Bh, n, max(1, r - p_over), r, tau * d["delta"])
    out = dict(X=torch.fft.irfft(Xh, n=n, dim=0), k=k, r=r)
    if full:
        out.update(Xh=Xh, V=V[:, :, :k], S=S[:, :k], U=Q @ UbH.mH[:, :, :k])
    return out


def _exact_ttsvd(d, tau):
    n = d["A"].shape[0]
    Ah, Bh = _hat(d["A"]), _hat(d["B"])
    U, S, VH = _svd(Ah)
    k, Xh = _truncated(VH.mH, S, U.mH @ Bh, Ah, Bh, n, 1, S.shape[1], tau * d["delta"])
    return dict(X=torch.fft.irfft(Xh, n=n, dim=0), k=k)


def _bidiagonalise(Ah, b, bound, k_max, n, k_fixed=None):
    """Golub-Kahan steps per Fourier slice with full reorthogonalisation, up to the first k whose projected
    residual meets the bound: W, the bidiagonal (c, z) and k."""
    w = _weights(n)
    project = lambda v, basis: v - (torch.stack(basis, -1) @ (torch.stack(basis, -1).mH @ v[..., None]))[..., 0]
    norm = lambda v: torch.sqrt((v.real ** 2 + v.imag ** 2).sum(-1))
    z = [norm(b)]
    Q, W, c = [b / z[0][:, None]], [], []
    phibar, rhobar = z[0], None
    for i in range(1, k_max + 1):
        v = (Ah.mH @ Q[-1][..., None])[..., 0]
        if W:
            v = v - z[-1][:, None] * W[-1]
            for _ in range(2):
                v = project(v, W)
        c.append(norm(v))
        W.append(v / c[-1][:, None])
        u = (Ah @ W[-1][..., None])[..., 0] - c[-1][:, None] * Q[-1]
        for _ in range(2):
            u = project(u, Q)
        z.append(norm(u))
        Q.append(u / z[-1][:, None])
        if k_fixed is None:
            rhobar = c[0] if i == 1 else -cs * c[-1]
            rho = torch.hypot(rhobar, z[-1])
            cs, sn = rhobar / rho, z[-1] / rho
            phibar = sn * phibar
            if math.sqrt(float((w * phibar ** 2).sum()) / n) <= bound:
                break
        elif i == k_fixed:
            break
    return torch.stack(W, -1), torch.stack(c, -1), torch.stack(z, -1), len(c)


def _projected(c, z, lam):
    """argmin ||P y - z_1 e_1||^2 + lam ||y||^2 per slice, P the (k+1) x k lower bidiagonal."""
    k = c.shape[1]
    P = torch.diag_embed(c)
    P = torch.cat([P, P.new_zeros((P.shape[0], 1, k))], 1)
    low = torch.diag_embed(z[:, 1:])
    P = P + torch.cat([low.new_zeros((low.shape[0], 1, k)), low], 1)
    if lam > 0.0:
        P = torch.cat([P, math.sqrt(lam) * torch.eye(k, dtype=P.dtype, device=P.device).expand(P.shape[0], k, k)], 1)
    rhs = torch.zeros(P.shape[:2], dtype=P.dtype, device=P.device)
    rhs = torch.cat([z[:, :1], rhs[:, 1:]], 1)
    q, r = torch.linalg.qr(P)
    return torch.linalg.solve_triangular(r, (q.mT @ rhs[..., None]), upper=True)[..., 0], P[:, :k + 1], rhs[:, :k + 1]


def _exact_tgkb(A, B, bound, k_max, k=None):
    """The tGKB solution and its k; with k given, differentiable in A and B."""
    n = A.shape[0]
    W, c, z, k = _bidiagonalise(_hat(A), _hat(B)[:, :, 0], bound, k_max, n, k)
    y, _, _ = _projected(c, z, 0.0)
    return torch.fft.irfft((W @ y[..., None].to(W.dtype)), n=n, dim=0), k


def _tikhonov_mu(c, z, bound, n):
    w = _weights(n)

    def above(t):
        y, P, rhs = _projected(c, z, 10.0 ** -t)
        res = ((P @ y[..., None])[..., 0] - rhs)
        return math.sqrt(float((w * (res ** 2).sum(-1)).sum()) / n) > bound

    lo, hi = math.log10(MU_LO), math.log10(MU_HI)
    if above(hi):
        return 10.0 ** hi
    if not above(lo):
        return 10.0 ** lo
    while hi - lo > 1e-11:
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if above(mid) else (lo, mid)
    return 10.0 ** hi


def _exact_tgkt(A, B, bound, k_max):
    n = A.shape[0]
    W, c, z, k = _bidiagonalise(_hat(A), _hat(B)[:, :, 0], bound, k_max, n)
    y, _, _ = _projected(c, z, 1.0 / _tikhonov_mu(c, z, bound, n))
    return torch.fft.irfft(W @ y[..., None].to(W.dtype), n=n, dim=0), k


def _exact_grad(case, d, G):
    n, bound = case["n"], case["tau"] * d["delta"]
    if case["method"] == "tgkb":
        with torch.no_grad():
            _, k = _exact_tgkb(d["A"], d["B"], bound, case["k_max"])
        c, B = d["c"].double().requires_grad_(), d["B"].double().requires_grad_()
        product = c[:, None, None] * d["T"].double()
        A = product + (d["A"].double() - product).detach()  # the float32 operator's values, c's derivative
        X, _ = _exact_tgkb(A, B, bound, case["k_max"], k)
        dB, dc = torch.autograd.grad(X, (B, c), G.double())
        return dict(X=X.detach(), dB=dB, dc=dc)
    f = _exact_rtsvd(d, case["tau"], case["p_over"], case["block"], case["r_max"], case["eps_rel"], full=True)
    Gh = _hat(G)
    dB = torch.fft.irfft(f["U"] @ ((f["V"].mH @ Gh) / f["S"][:, :, None]), n=n, dim=0)
    # X-hat_s = M_s B-hat_s / c-hat_s for A(:,:,k) = c_k T
    ch = torch.fft.rfft(d["c"].double())
    g = _weights(n) * (Gh.conj() * f["Xh"]).sum((1, 2)) / ch
    s, k = (torch.arange(m, dtype=torch.float64, device=DEVICE) for m in (n // 2 + 1, n))
    turn = torch.exp(-2j * math.pi / n * torch.remainder(k[:, None] * s, n))
    return dict(X=f["X"], dB=dB, dc=-(turn @ g).real / n)


def exact(case, seed):
    op = case["op"]
    if op in ("product", "product_grad"):
        st = prepare(case, seed)
        A, B = _hat(st["A"].detach()), _hat(st["B"].detach())
        back = lambda v: torch.fft.irfft(v, n=case["n"], dim=0)
        if op == "product":
            return back(A @ B)
        G = _hat(st["G"])
        return dict(C=back(A @ B), dA=back(G @ B.mH), dB=back(A.mH @ G))
    if op == "spectrum":
        A = prepare(case, seed)["A"].double()
        return dict(spectrum=torch.fft.rfft(A, dim=0), back=A)
    if op == "batch":
        out = []
        for d in _problems(case, seed):
            f = _exact_rtsvd(d, case["tau"], synth.UNEVEN_P_OVER, synth.UNEVEN_BLOCK, d["Omega"].shape[2],
                             d["eps_rel"])
            out.append(dict(rtsvd=f["X"], tgkb=_exact_tgkb(d["A"], d["B"], case["tau"] * d["delta"], d["k_max"])[0]))
        return out
    d = _problem(case, seed, case["N"], case["n"], case.get("p", 1), case.get("r_max", 0))
    bound = case["tau"] * d["delta"]
    if op == "rtsvd":
        f = _exact_rtsvd(d, case["tau"], case["p_over"], case["block"], case["r_max"], case["eps_rel"])
        return dict(X=f["X"], k=f["k"], r=f["r"])
    if op == "tgkt":
        X, k = _exact_tgkt(d["A"], d["B"], bound, case["k_max"])
        return dict(X=X, k=k)
    if op == "tgkb":
        bounds = d["deltas"] if case["p"] > 1 else [d["delta"]]
        got = [_exact_tgkb(d["A"], d["B"][:, :, j:j + 1], case["tau"] * b, case["k_max"])
               for j, b in enumerate(bounds)]
        return dict(X=torch.cat([X for X, _ in got], 2), k=[k for _, k in got])
    if op == "ttsvd":
        return _exact_ttsvd(d, case["tau"])
    if op == "plain":
        t = _exact_ttsvd(d, case["tau"])
        f = _exact_rtsvd(d, case["tau"], case["p_over"], case["block"], case["r_max"], case["eps_rel"])
        X, k = _exact_tgkb(d["A"], d["B"], bound, case["k_max"])
        return dict(ttsvd=t["X"], rtsvd=f["X"], tgkb=X, k=[t["k"], f["k"], k])
    return _exact_grad(case, d, _cotangent(case, seed))
