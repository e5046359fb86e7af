"""Performance cases: what programs have this library do, through its public entry points.

The library's path is the polar factorisation A = U H by the Newton-Schulz iteration, so most cases are
solves, from a single small matrix (where latency and launches count) to the largest one that is solved
many times in a row; the rest are the entry points built on the same kernels: batched solves, products,
the Newton-Schulz inverse and the Chebyshev matrix function. Sizes come from this repository's workloads,
tests and benchmark (512^2 kappa 1e2, 8192^2 kappa 1e4, 1000 x 700, the 4:1 tall shape, the batched size
law, degree-32 Chebyshev series) or are generic and ragged.

Inputs are dense matrices with a prescribed singular spectrum (log-spaced, as in the package's synthetic
workloads), A = Q1 diag(sigma) Q2^T, with Q1 and Q2 sign-scrambled cosine bases instead of Haar factors:
they are drawn in milliseconds at every size, and A is dense with entries of comparable magnitude.
"""
from __future__ import annotations

import math

import torch

from paper_2112_09017_gb300 import polar, synth

DEV = "cuda"

# ------------------------------------------------------------------------------------------ the cases


def listed():
    return [
        # one small matrix between other work of a program: a frame of directions, a small layer's update;
        # the time is launches and latency
        {"name": "solve_96x64", "kind": "solve", "m": 96, "n": 64, "kappa": 1e2, "prec": "bf16x6", "pre": False},
        # precision left to the library at a size where it picks plain float32
        {"name": "solve_auto_300x200", "kind": "solve", "m": 300, "n": 200, "kappa": 1e3, "prec": "auto", "pre": False},
        # the repository's 512^2 workload in the default precision
        {"name": "solve_512", "kind": "solve", "m": 512, "n": 512, "kappa": 1e2, "prec": "bf16x6", "pre": False},
        # an odd-sized tall matrix (tests): remainders in every tile direction
        {"name": "solve_1000x700", "kind": "solve", "m": 1000, "n": 700, "kappa": 1e3, "prec": "bf16x6", "pre": False},
        # a hidden-size weight matrix with the preconditioned iteration (Algorithm 1)
        {"name": "solve_2048_pre", "kind": "solve", "m": 2048, "n": 2048, "kappa": 1e4, "prec": "bf16x6", "pre": True},
        # the tall workload's 4:1 shape and conditioning, scaled down
        {"name": "solve_8192x2048", "kind": "solve", "m": 8192, "n": 2048, "kappa": 1e6, "prec": "bf16x6", "pre": False},
        # the repository's 8192^2 workload: the largest case
        {"name": "solve_8192", "kind": "solve", "m": 8192, "n": 8192, "kappa": 1e4, "prec": "bf16x6", "pre": False},
        # uneven problems in one call (the batched configuration's size law, a 256-problem batch)
        {"name": "batched_256", "kind": "batched", "count": 256, "n_lo": 64, "n_hi": 1024, "kappa": 1e3, "sizes": 0},
        # many small problems in one call (the benchmark's small batch, n on [64, 128])
        {"name": "batched_small_1024", "kind": "batched", "count": 1024, "n_lo": 64, "n_hi": 128, "kappa": 1e3,
         "sizes": 1},
        # a float32-grade product of ragged matrices with a transposed operand
        {"name": "gemm_3000x2500x4000_t", "kind": "gemm", "M": 3000, "N": 2500, "K": 4000, "ta": True, "tb": False,
         "prec": "bf16x6"},
        # Newton-Schulz inverse of a well-conditioned odd-sized matrix
        {"name": "inverse_1001", "kind": "inverse", "m": 1001, "n": 1001, "kappa": 10.0},
        # exp(A) of a symmetric matrix by the benchmark's degree-32 Chebyshev series
        {"name": "chebyshev_1536_d32", "kind": "cheb", "n": 1536, "degree": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["batched"] * 2 + ["gemm", "inverse", "cheb"])
    if kind == "solve":
        prec = rng.choice(["bf16x6"] * 6 + ["auto", "fp32"])
        n = _log_int(rng, 24, 512 if prec == "fp32" else 4096)
        m = n if rng.random() < 0.4 else int(n * rng.uniform(1.0, 4.0))
        return {"kind": "solve", "m": m, "n": n, "kappa": float(round(10.0 ** rng.uniform(1.0, 4.0), 1)), "prec": prec,
                "pre": rng.random() < 0.2}
    if kind == "batched":
        if rng.random() < 0.5:
            return {"kind": "batched", "count": _log_int(rng, 16, 256), "n_lo": 64, "n_hi": 1024, "kappa": 1e3,
                    "sizes": rng.randrange(2, 10 ** 6)}
        return {"kind": "batched", "count": _log_int(rng, 64, 2048), "n_lo": 16, "n_hi": 128, "kappa": 1e3,
                "sizes": rng.randrange(2, 10 ** 6)}
    if kind == "gemm":
        return {"kind": "gemm", "M": _log_int(rng, 48, 6000), "N": _log_int(rng, 48, 6000), "K": _log_int(rng, 48, 6000),
                "ta": rng.random() < 0.5, "tb": rng.random() < 0.5, "prec": rng.choice(["bf16x6", "auto"])}
    if kind == "inverse":
        n = _log_int(rng, 32, 2500)
        m = n if rng.random() < 0.6 else int(n * rng.uniform(1.0, 2.0))
        return {"kind": "inverse", "m": m, "n": n, "kappa": float(round(rng.uniform(2.0, 12.0), 1))}
    return {"kind": "cheb", "n": _log_int(rng, 32, 3000), "degree": rng.randrange(6, 41)}


# ------------------------------------------------------------------------------------------ inputs


def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + salt * 7919 + 12345) % (2 ** 62))


def _signs(n, g, dt):
    return torch.randint(0, 2, (n,), generator=g, device=DEV).to(dt).mul_(2).sub_(1)


def _cos_basis(m, n, g, dt):
    """m x n with orthonormal columns: n columns of the orthogonal cosine basis, rows sign-scrambled."""
    i = (torch.arange(m, device=DEV, dtype=torch.float64) + 0.5)[:, None]
    j = torch.arange(n, device=DEV, dtype=torch.float64)[None, :]
    q = torch.cos(i * j * (math.pi / m)).mul_(math.sqrt(2.0 / m))
    q[:, 0] = math.sqrt(1.0 / m)
    return (q * _signs(m, g, torch.float64)[:, None]).to(dt)


def _spectral_matrix(m, n, kappa, g):
    dt = torch.float64 if m * n <= 2 ** 22 else torch.float32   # the product's precision; the large kappas are below
    if kappa > 1e5:
        dt = torch.float64                                      # float32's rounding would bury the spectrum's low end
    s = torch.from_numpy(synth.logspace_spectrum(n, 1.0 / kappa)).to(device=DEV, dtype=dt)
    s = s[torch.randperm(n, generator=g, device=DEV)]
    return ((_cos_basis(m, n, g, dt) * s[None, :]) @ _cos_basis(n, n, g, dt).T).to(torch.float32).contiguous()


def _symmetric_matrix(n, g):
    q = _cos_basis(n, n, g, torch.float64)
    lam = torch.linspace(-1.0, 1.0, n, device=DEV, dtype=torch.float64)[torch.randperm(n, generator=g, device=DEV)]
    a = (q * lam[None, :]) @ q.T
    return (0.5 * (a + a.T)).to(torch.float32).contiguous()


def _batch_sizes(case):
    """The batched size law: n uniform, m = n or 2 n; fixed by the case, as a program's plan is."""
    import numpy as np
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        out.append((n if rng.random() < 0.5 else 2 * n, n))
    return out


def _inputs(case, seed):
    g = _gen(seed)
    k = case["kind"]
    if k in ("solve", "inverse"):
        return [_spectral_matrix(case["m"], case["n"], case["kappa"], g)]
    if k == "batched":
        return [_spectral_matrix(m, n, case["kappa"], g) for m, n in _batch_sizes(case)]
    if k == "gemm":
        sa = (case["K"], case["M"]) if case["ta"] else (case["M"], case["K"])
        sb = (case["N"], case["K"]) if case["tb"] else (case["K"], case["N"])
        return [torch.randn(s, generator=g, device=DEV) for s in (sa, sb)]
    return [_symmetric_matrix(case["n"], g)]


def _packed(shapes, dtype=torch.float32):
    """One zeroed buffer and a view of it for each shape, each starting on a multiple of 64 elements."""
    starts, total = [], 0
    for r, c in shapes:
        starts.append(total)
        total += (r * c + 63) // 64 * 64
    buf = torch.zeros((total,), dtype=dtype, device=DEV)
    return buf, [buf[o:o + r * c].view(r, c) for o, (r, c) in zip(starts, shapes)]


class _Batched:
    """A batched plan that is destroyed with its owner."""

    def __init__(self, sizes):
        self.plan = polar.polar_batched_plan_create([m for m, _ in sizes], [n for _, n in sizes])

    def __del__(self):
        polar.polar_plan_destroy(self.plan)


def prepare(case, seed):
    k = case["kind"]
    x = _inputs(case, seed)
    st = {"case": case, "x": x}
    if k == "solve":
        m, n = case["m"], case["n"]
        st["plan"] = polar.Plan(m, n, prec=case["prec"], precondition=int(case["pre"]))
        st["U"] = torch.empty((m, n), device=DEV)
        st["H"] = torch.empty((n, n), device=DEV)
    elif k == "batched":
        st["owner"] = _Batched([tuple(a.shape) for a in x])
        # every U in one buffer and every H in another, each problem's matrix packed in its own part
        st["U"], u = _packed([tuple(a.shape) for a in x])
        st["H"], h = _packed([(a.shape[1], a.shape[1]) for a in x])
        st["bound"] = polar.polar_batched_bind(st["owner"].plan, x, u, h)
    elif k == "gemm":
        st["C"] = torch.empty((case["M"], case["N"]), device=DEV)
    elif k == "inverse":
        st["X"] = torch.empty((case["n"], case["m"]), device=DEV)
    else:
        st["F"] = torch.empty_like(x[0])
        st["coef"] = polar.chebyshev_coefficients(math.exp, -1.0, 1.0, case["degree"])
    return st


# ------------------------------------------------------------------------------------------ one pass


def run(st):
    case, x = st["case"], st["x"]
    k = case["kind"]
    if k == "solve":
        st["plan"](x[0], U=st["U"], H=st["H"])
        return {"U": st["U"], "H": st["H"]}
    if k == "batched":
        polar.polar_batched_run(st["owner"].plan, st["bound"])
        return {"U": st["U"], "H": st["H"]}
    if k == "gemm":
        polar.polar_gemm(x[0], x[1], st["C"], case["ta"], case["tb"], prec=polar.PREC[case["prec"]])
        return st["C"]
    if k == "inverse":
        polar.polar_ns_inverse(x[0], st["X"])
        return st["X"]
    polar.polar_chebyshev(x[0], st["F"], -1.0, 1.0, st["coef"])
    return st["F"]


# ------------------------------------------------------------------------------------------ work


def _updates(n, fnorm2, sigma, pre):
    """Updates the iteration applies to a matrix with these singular values (the scalar recurrence)."""
    s = [v / math.sqrt(fnorm2) for v in sigma]
    k = 0
    if pre:
        a = 1.5 * math.sqrt(3.0) - 0.1
        low = 2.0 ** -23
        while low < 0.1:
            low = a * low * (1.0 - (4.0 / 27.0) * a * a * low * low)
            s = [a * v * (1.0 - (4.0 / 27.0) * a * a * v * v) for v in s]
            k += 1
    while k < 100 and math.sqrt(sum((v * v - 1.0) ** 2 for v in s) / n) > 1e-6:
        s = [0.5 * v * (3.0 - v * v) for v in s]
        k += 1
    return k


def _solve_flops(m, n, kappa, pre):
    sigma = synth.logspace_spectrum(n, 1.0 / kappa)
    sigma = sigma if n <= 256 else sigma[:: max(1, n // 256)]
    k = _updates(len(sigma), float((sigma ** 2).sum()) * n / len(sigma), sigma.tolist(), pre)
    # k + 1 Gram triangles of m n^2, k updates of 2 m n^2, U^T A of 2 m n^2
    return float(m) * n * n * (3 * k + 3)


def work(case):
    k = case["kind"]
    if k == "solve":
        m, n = case["m"], case["n"]
        return {"bytes": 4 * (2 * m * n + n * n), "flops": _solve_flops(m, n, case["kappa"], case["pre"])}
    if k == "batched":
        sizes = _batch_sizes(case)
        per = {}
        f = 0.0
        for m, n in sizes:
            if n not in per:
                per[n] = _solve_flops(1, n, case["kappa"], False)
            f += m * per[n]
        return {"bytes": sum(4 * (2 * m * n + n * n) for m, n in sizes), "flops": f}
    if k == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * (M * K + K * N + M * N), "flops": 2.0 * M * N * K}
    if k == "inverse":
        m, n = case["m"], case["n"]
        # the Gram triangle for the scaling, then A X and X P for each of about 4 + 2 log2(kappa) + 4 updates
        it = 8 + int(2 * math.log2(max(2.0, case["kappa"])))
        return {"bytes": 4 * 2 * m * n, "flops": float(m) * n * n + it * 4.0 * m * m * n}
    n, d = case["n"], case["degree"]
    return {"bytes": 4 * (n * (n + 1) // 2 + n * n), "flops": float(d - 1) * n ** 3}   # triangles of symmetric products


# ------------------------------------------------------------------------------------------ correctness


def tolerance(case):
    k = case["kind"]
    if k in ("solve", "batched"):
        # U moves by about 2^-24 kappa in its least singular directions; measured against float64: 7e-7 at 96 x 64
        # and kappa 1e2, 4.7e-6 at 1000 x 700 and 1e3, 3.5e-3 at 8192 x 2048 and 1e6 (H: 1e-7 to 4e-7)
        n = case["n"] if k == "solve" else case["n_lo"]
        return {"rel": max(3e-6, case["kappa"] * (1e-8 + 1.5e-7 / math.sqrt(n)))}
    if k == "gemm":
        return {"rel": 1.4e-6}                               # measured 3.5e-7
    if k == "inverse":
        return {"rel": max(1.2e-6, 1.5e-7 * case["kappa"])}  # measured 3.1e-7 at kappa 10
    return {"rel": 1.2e-6}                                   # measured 2.1e-7


def _polar64(a):
    """Polar factors of a stack of float64 matrices (b, m, n): QR, then Newton's iteration with Higham's
    scaling on the triangular factor."""
    q, x = torch.linalg.qr(a)
    n = x.shape[-1]
    for _ in range(60):
        y = torch.linalg.inv(x).mT
        nx = torch.linalg.matrix_norm(x)[:, None, None]
        g = torch.sqrt(torch.linalg.matrix_norm(y)[:, None, None] / nx)
        close = (nx * nx / n - 1.0).abs() < 1e-2
        g = torch.where(close, torch.ones_like(g), g)
        xn = 0.5 * (g * x + y / g)
        done = bool((torch.linalg.matrix_norm(xn - x)[:, None, None] <= 1e-13 * nx).all())
        x = xn
        if done:
            break
    u = q @ x
    h = u.mT @ a
    return u, 0.5 * (h + h.mT)


def _inverse64(a):
    """Algorithm 2 in float64: X <- X (2 I - A X) from A^T / ||A A^T||_F until the relative step is below
    2^(k - 24) after update k."""
    x = a.T / torch.linalg.matrix_norm(a.T @ a)
    for k in range(100):
        xn = 2.0 * x - x @ (a @ x)
        step = float(torch.linalg.matrix_norm(xn - x) / torch.linalg.matrix_norm(xn))
        x = xn
        if step <= 2.0 ** (k - 24):
            break
    return x


def exact(case, seed):
    k = case["kind"]
    x = _inputs(case, seed)
    if k == "solve":
        if case["m"] * float(case["n"]) ** 2 > 1.5e11:
            return None                                  # minutes in float64 on this hardware
        u, h = _polar64(x[0].double()[None])
        return {"U": u[0], "H": h[0]}
    if k == "batched":
        out_u, us = _packed([tuple(a.shape) for a in x], torch.float64)
        out_h, hs = _packed([(a.shape[1], a.shape[1]) for a in x], torch.float64)
        groups = {}
        for i, a in enumerate(x):
            groups.setdefault(tuple(a.shape), []).append(i)
        for idx in groups.values():
            u, h = _polar64(torch.stack([x[i] for i in idx]).double())
            for t, i in enumerate(idx):
                us[i].copy_(u[t])
                hs[i].copy_(h[t])
        return {"U": out_u, "H": out_h}
    if k == "gemm":
        a = (x[0].T if case["ta"] else x[0]).double()
        b = (x[1].T if case["tb"] else x[1]).double()
        return a @ b
    if k == "inverse":
        return _inverse64(x[0].double())
    lam, q = torch.linalg.eigh(x[0].double())
    # the interpolant of exp through the degree + 1 first-kind Chebyshev points, at the eigenvalues
    d = case["degree"]
    th = math.pi * (torch.arange(d + 1, dtype=torch.float64, device=DEV) + 0.5) / (d + 1)
    g = torch.exp(torch.cos(th))
    c = 2.0 / (d + 1) * (torch.cos(torch.arange(d + 1, dtype=torch.float64, device=DEV)[:, None] * th[None, :]) @ g)
    c[0] *= 0.5
    b1, b2 = torch.zeros_like(lam), torch.zeros_like(lam)
    for j in range(d, 0, -1):
        b1, b2 = c[j] + 2.0 * lam * b1 - b2, b1
    p = c[0] + lam * b1 - b2
    return (q * p[None, :]) @ q.T
