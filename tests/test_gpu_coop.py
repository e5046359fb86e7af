"""The single solve in one cooperative launch (three planes, small and medium sizes): parity with the
float64 oracle at the edges of its tiles and of its dispatch, agreement with the separate launches, and
its statuses."""
import math

import numpy as np
import pytest

from oracle.ns_polar import ns_polar
from paper_2112_09017_gb300 import synth

from .gpu_util import metrics, to_np

pytestmark = pytest.mark.gpu


def _solve(lib, a, prec="bf16x6", **kw):
    import torch
    m, n = a.shape
    plan = lib.Plan(m, n, prec=prec, **kw)
    U, H, info = plan(torch.from_numpy(a).cuda(), raw_status=True)
    plan.close()
    return to_np(U), to_np(H), info


# one tile, tile edges in rows (128) and columns (64 and 128), an odd and an even number of 64-wide columns
# (the triangle's pairs), k-block remainders, tall and narrow, tiles shared by four and by two blocks and by
# none (parts of K that are empty among them), whole tiles of either width, more tiles than SMs, the
# tallest size of one launch and one row more
SIZES = [(1, 1), (32, 31), (64, 64), (128, 65), (129, 128), (130, 129), (192, 192), (257, 200), (384, 320),
         (2500, 33), (700, 700), (740, 740), (1000, 700), (1000, 996), (1300, 1290), (1744, 1312), (2100, 2050),
         (2400, 2304), (155648, 33), (155649, 33)]


# the plain form's 32 x 32 tiles: edges, remainders of the 64-deep chunks, near the largest square one, and beyond it
SIZES32 = [(1, 1), (31, 31), (33, 32), (64, 33), (65, 64), (300, 200), (130, 129), (3000, 40), (1000, 990),
           (1640, 1640), (1700, 1650), (2000, 2000)]
SEPARATE = [("bf16x6", 155649, 33), ("fp32", 1700, 1650), ("fp32", 2000, 2000)]


@pytest.mark.parametrize("prec,m,n", [("bf16x6", *s) for s in SIZES] + [("fp32", *s) for s in SIZES32],
                         ids=lambda v: str(v))
def test_coop_solve_matches_oracle_and_separate_launches(lib, prec, m, n):
    kappa = 50.0
    a = synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 1.0 / kappa), 40 + n)
    U, H, info = _solve(lib, a, prec)
    # a residual history that may not hold every step sends a plan to the separate launches
    U2, H2, info2 = _solve(lib, a, prec, max_iter=lib.POLAR_HIST + 10)
    assert info["status"] == info2["status"] == lib.POLAR_OK
    # G's diagonal is a float32 sum over the rows: with 155648 its rounding is of the size of the tolerance
    assert abs(info["iters"] - info2["iters"]) <= (m > 100000), (info["res_hist"][-3:], info2["res_hist"][-3:])
    assert (info["launches"] > 1) == ((prec, m, n) in SEPARATE) and info2["launches"] > 1
    # the residuals differ by the rounding of G: about 1e-6 of them far from convergence
    for g, w in zip(info["res_hist"], info2["res_hist"]):
        if w > 1e-3:
            assert abs(g - w) <= 1e-4 * w
    assert info["sym_err"] <= 1e-5 and abs(info["normA_F"] - info2["normA_F"]) <= 1e-12 * info["normA_F"]
    # each is within the forward bound 1e-7 kappa of the exact factor
    assert np.linalg.norm(U.astype(np.float64) - U2) / math.sqrt(n) <= 2e-7 * kappa
    ref = ns_polar(a, tol=1e-12, count_tol=1e-6) if n <= 1300 and m < 155648 else None
    met = metrics(a, U, H, ref["U"] if ref else None)
    assert met["orth"] <= 5e-6 and met["bwd"] <= 5e-6 and met["hsym"] == 0.0, met
    if ref:
        assert abs(info["iters"] - ref["iters_at"]) <= 1
        assert met["fwd"] <= 1e-7 * kappa, met


@pytest.mark.parametrize("prec", ["bf16x6", "fp32"])
def test_coop_statuses_and_reuse(lib, prec):
    """Zero and non-finite input leave U and H untouched, max_iter returns the last iterate, and the same
    plan solves again afterwards, bit for bit the same twice."""
    import torch
    m, n = 300, 260
    a = torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 1e-2), 3)).cuda()
    plan = lib.Plan(m, n, prec=prec, max_iter=20)
    U = torch.full((m, n), 7.0, device="cuda")
    H = torch.full((n, n), 7.0, device="cuda")
    bad = a.clone()
    bad[17, 5] = float("nan")
    for x in (torch.zeros_like(a), bad, torch.full_like(a, float("inf"))):
        _, _, info = plan(x, U=U, H=H, raw_status=True)
        assert info["status"] == lib.POLAR_ENONFINITE
        assert bool(torch.all(U == 7.0)) and bool(torch.all(H == 7.0))
    U1, H1, i1 = plan(a)
    U2, H2, i2 = plan(a)
    assert i1["status"] == lib.POLAR_OK and i1["res_hist"] == i2["res_hist"]
    assert torch.equal(U1, U2) and torch.equal(H1, H2)
    plan.close()
    plan = lib.Plan(m, n, prec=prec, max_iter=5)
    U3, H3, i3 = plan(a, raw_status=True)
    plan.close()
    assert i3["status"] == lib.POLAR_NOT_CONVERGED and i3["iters"] == 5 and len(i3["res_hist"]) == 6
    assert i3["res_hist"] == i1["res_hist"][:6]
    assert bool(torch.isfinite(U3).all()) and bool(torch.isfinite(H3).all())


def _four_squares(r):
    """Four integers whose squares sum to r."""
    for a in range(math.isqrt(r), -1, -1):
        for b in range(min(a, math.isqrt(r - a * a)), -1, -1):
            s = r - a * a - b * b
            for c in range(min(b, math.isqrt(s)), -1, -1):
                d = math.isqrt(s - c * c)
                if c * c + d * d == s:
                    return a, b, c, d
    raise AssertionError


def _exact_residual_matrix(n, k, seed):
    """A with ||A||_F = 2^k to float32, whose first Gram matrix has entries that float32 holds exactly and at most
    one besides the zeros in 32 consecutive columns of a row, and v = ||G - I||_F^2 of these entries with every
    square rounded to float32, as an exact fraction: the first n / 2 columns hold integers below 2^8 on the
    diagonal, the others 2^-14 times such integers, n / 2 rows up."""
    from fractions import Fraction
    rng = np.random.default_rng(seed)
    h = n // 2
    mean = 2.0 ** k / math.sqrt(h)
    d = rng.integers(int(0.6 * mean), int(1.3 * mean), h).astype(np.int64)
    left, i = 4 ** k - int((d[:h - 4] ** 2).sum()), 0
    while not 0 <= left <= 8 * mean ** 2:          # to within four more entries
        step = 1 if left > 0 else -1
        left -= 2 * step * int(d[i]) + 1
        d[i] += step
        i = (i + 1) % (h - 4)
    d[h - 4:] = _four_squares(left)
    assert 0 <= d.min() and d.max() < 256 and (d ** 2).sum() == 4 ** k
    a = np.zeros((n, n))
    i = np.arange(h)
    a[i, i] = d
    a[i, i + h] = rng.integers(1, 256, h) * 2.0 ** -14
    assert np.float32(np.linalg.norm(a)) == 2.0 ** k
    x = a / 2.0 ** k
    dev = np.float32((x ** 2).sum(0)) - np.float32(1.0)
    off = np.float32(x[i, i] * x[i, i + h])
    v = sum((Fraction(float(t)) for t in dev * dev), Fraction(0))
    return a.astype(np.float32), v + 2 * sum((Fraction(float(t)) for t in off * off), Fraction(0))


# one block, tiles shared by four blocks, whole tiles in one wave and in three, one SM of a batch, the batch's tiles
@pytest.mark.parametrize("n,k,how", [(96, 9, "solve"), (512, 10, "solve"), (1300, 11, "solve"), (2304, 11, "solve"),
                                     (96, 9, "batch"), (512, 10, "batch")], ids=lambda v: str(v))
def test_residuals_are_summed_in_float64(lib, n, k, how):
    """The reported residual of the first step against the exact sum of its float32 terms. At most 40 float64
    additions one after another, each off by 0.58 * 2^-53 at the most in the mean, come to 2.0e-16 halved by the
    square root, with the roundings of that and of the scaling 1.2e-16 in all; measured 0.5e-16 to 1.3e-16, and
    4.4e-16 to 1.4e-15 with pairs of floats."""
    import torch
    errs = []
    for seed in range(6):
        a, v = _exact_residual_matrix(n, k, 10 * seed + n)
        t = torch.from_numpy(a).cuda()
        want = math.sqrt(float(v)) / math.sqrt(n)
        if how == "solve":
            plan = lib.Plan(n, n)
            _, _, info = plan(t, tol=2.0)              # stops at X_0
            plan.close()
            assert info["iters"] == 0
            got = info["res_hist"][0]
        else:
            plan = lib.polar_batched_plan_create([n], [n])
            r = torch.zeros(1, dtype=torch.float64, device="cuda")
            lib.polar_batched_run(plan, [t], [torch.empty_like(t)], [torch.empty_like(t)], 2.0, None, r)
            got = float(r[0])
            lib.polar_plan_destroy(plan)
        errs.append((got - want) / want)
    assert np.sqrt(np.mean(np.square(errs))) <= 3e-16, errs


@pytest.mark.parametrize("prec,m,n,seeds", [("bf16x6", 8, 8, 12), ("bf16x6", 96, 64, 12), ("fp32", 300, 200, 12),
                                            ("bf16x6", 3000, 2900, 3), ("bf16x6", 5000, 4500, 2)], ids=lambda v: str(v))
def test_norm_is_summed_in_float64(lib, prec, m, n, seeds):
    """||A||_F against the exact sum of squares, entries over eleven binades. A float64 sum as the kernels order it
    (at most some 40 additions one after another) is off by about 1e-16, as in the test of the residuals; pairs
    of floats by 3e-16 to 7.6e-16."""
    import torch
    plan = lib.Plan(m, n, prec=prec, max_iter=1)
    errs = []
    for seed in range(seeds):
        rng = np.random.default_rng(1000 * seed + m + n)
        a = (rng.standard_normal((m, n)) * 2.0 ** rng.integers(-5, 6, (m, n))).astype(np.float32)
        want = math.sqrt(math.fsum((a.astype(np.float64) ** 2).reshape(-1)))   # the squares are exact
        _, _, info = plan(torch.from_numpy(a).cuda(), raw_status=True)
        errs.append((info["normA_F"] - want) / want)
    plan.close()
    assert np.sqrt(np.mean(np.square(errs))) <= 2.5e-16, errs


PLAIN = [(31, 33, 1, 0), (32, 64, 64, 0), (100, 700, 130, 1), (700, 40, 129, 0), (900, 600, 520, 1)]


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("M,N,K,off", PLAIN, ids=lambda v: str(v))
def test_fp32_products_in_small_tiles(lib, ta, tb, M, N, K, off):
    """Both storage orders of both operands, tile and chunk remainders, aligned rows and rows that are not
    (a view one element into a wider matrix), with C read and written in place."""
    import torch

    from .gpu_util import gemm_bound
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((K, M) if ta else (M, K)).astype(np.float32)
    b = rng.standard_normal((N, K) if tb else (K, N)).astype(np.float32)
    c = rng.standard_normal((M, N)).astype(np.float32)

    def view(x):
        big = torch.full((x.shape[0] + 1, x.shape[1] + 3 * off), float("nan"), device="cuda")
        v = big[:x.shape[0], off:off + x.shape[1]]
        v.copy_(torch.from_numpy(x))
        return v

    C = torch.from_numpy(c).cuda()
    lib.polar_gemm(view(a), view(b), C, ta, tb, 0.75, -1.25, lib.POLAR_FP32)
    A64 = (a.T if ta else a).astype(np.float64)
    B64 = (b.T if tb else b).astype(np.float64)
    err = np.abs(to_np(C).astype(np.float64) - (0.75 * A64 @ B64 - 1.25 * c.astype(np.float64)))
    assert np.all(err <= gemm_bound(np.abs(A64), np.abs(B64), K, np.abs(c), 0.75, -1.25))


# tiles shared by four blocks and by two, whole tiles in one wave and in two, and 128 x 256 tiles; C's rows aligned and
# not (a view one element into a wider matrix)
GEMMS = [(48, 70, 6000, 0), (129, 65, 200, 1), (400, 640, 700, 1), (700, 500, 260, 1), (1000, 1001, 97, 0),
         (1500, 1400, 300, 1), (2000, 1500, 131, 1)]


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("M,N,K,off", GEMMS, ids=lambda v: str(v))
def test_bf16x6_products_in_narrow_tiles(lib, ta, tb, M, N, K, off):
    import torch

    from .gpu_util import gemm_bound
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((K, M) if ta else (M, K)).astype(np.float32)
    b = rng.standard_normal((N, K) if tb else (K, N)).astype(np.float32)
    c = rng.standard_normal((M, N)).astype(np.float32)
    big = torch.full((M + 1, N + 3 * off), 7.0, device="cuda")
    C = big[:M, off:off + N]
    for beta in (-1.25, 0.0):
        C.copy_(torch.from_numpy(c) if beta else torch.full((M, N), float("nan")))
        lib.polar_gemm(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), C, ta, tb, 0.75, beta, lib.POLAR_BF16X6)
        A64 = (a.T if ta else a).astype(np.float64)
        B64 = (b.T if tb else b).astype(np.float64)
        err = np.abs(to_np(C).astype(np.float64) - (0.75 * A64 @ B64 + beta * c.astype(np.float64)))
        assert np.all(err <= gemm_bound(np.abs(A64), np.abs(B64), K, np.abs(c), 0.75, beta, 3))
        C.fill_(7.0)
        assert bool((big == 7.0).all())   # nothing beside C was written


# sizes of the inverse's and the Chebyshev function's dispatch and tiles that their own tests do not reach: tiles
# shared by two blocks, 64- and 128-wide ones over the whole chip, more than a wave
INVERSES = [(520, 390), (700, 700), (1001, 1001), (1300, 1250), (2100, 700), (2400, 2300)]


@pytest.mark.parametrize("m,n", INVERSES, ids=lambda v: str(v))
def test_coop_inverse_matches_separate_launches(lib, monkeypatch, m, n):
    import torch
    a = torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 0.2), m)).cuda()
    big = torch.full((n + 2, m + 7), 9.0, device="cuda")
    X = big[1:n + 1, 3:m + 3]                       # strided, unaligned rows
    out = lib.polar_ns_inverse(a, X)
    monkeypatch.setenv("POLAR_TC_CTA_PAIR", "0")    # names a form: the separate launches
    Y = torch.empty((n, m), device="cuda")
    ref = lib.polar_ns_inverse(a, Y)
    assert out["status"] == ref["status"] == lib.POLAR_OK and out["iters"] == ref["iters"]
    # delta is a ratio of rounded sums over the last, small step
    assert out["delta"] == pytest.approx(ref["delta"], rel=1e-2, abs=1e-7)
    assert float(torch.linalg.matrix_norm(X - Y) / torch.linalg.matrix_norm(Y)) <= 2e-6
    xa = X.double() @ a.double()
    assert float(torch.linalg.matrix_norm(xa - torch.eye(n, device="cuda", dtype=torch.float64))) <= 1e-5 * math.sqrt(n)
    X.fill_(9.0)
    assert bool(torch.all(big == 9.0))


# tiles shared along K, whole tiles 64 and 128 wide in one launch, separate launches; the scales put ||X||_F between 3e19 and 5e19
@pytest.mark.parametrize("m,n,e,form", [(300, 300, -59, ""), (1001, 1001, -58, ""), (2400, 2300, -57, ""),
                                        (1001, 1001, -58, "0")], ids=lambda v: str(v))
def test_inverse_of_a_matrix_of_very_small_norm(lib, monkeypatch, m, n, e, form):
    """||X||_F^2 beyond float32's range, every entry's square and every sum of a row chunk well inside it: the
    relative steps, the updates and the result are those of the same matrix at unit scale."""
    import torch
    monkeypatch.setenv("POLAR_TC_CTA_PAIR", form)
    a = torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 0.1), m)).cuda()
    X, Y = torch.empty((n, m), device="cuda"), torch.empty((n, m), device="cuda")
    one = lib.polar_ns_inverse(a, X)
    tiny = lib.polar_ns_inverse(a * 2.0 ** e, Y, raw_status=True)
    assert float(torch.linalg.matrix_norm(Y.double())) > 2.0 ** 64
    assert tiny["status"] == one["status"] == lib.POLAR_OK
    assert tiny["iters"] == one["iters"] and tiny["delta"] == pytest.approx(one["delta"], rel=1e-2, abs=1e-7)
    # ||A^T A||_F of the tiny matrix is a sum of float32 denormals in part: another scale of X_0, another rounding
    assert float(torch.linalg.matrix_norm(Y * 2.0 ** e - X) / torch.linalg.matrix_norm(X)) <= 1e-5


@pytest.mark.parametrize("n", [100, 300, 640])
def test_inverse_in_cta_pairs_with_an_odd_row_of_tiles(lib, monkeypatch, n):
    """A pair whose second half lies past the last row still writes residual sums of its own; they have a
    place in the workspace (they once landed in the state after it, and the call reported an expired wait)."""
    import torch
    a = torch.from_numpy(synth.matrix_with_spectrum(n, n, synth.logspace_spectrum(n, 0.2), n)).cuda()
    out = []
    for form in ("0", "1"):
        monkeypatch.setenv("POLAR_TC_CTA_PAIR", form)
        X = torch.empty((n, n), device="cuda")
        out.append((lib.polar_ns_inverse(a, X), X))
    (i0, X0), (i1, X1) = out
    assert i0["status"] == i1["status"] == lib.POLAR_OK and i0["iters"] == i1["iters"]
    assert float(torch.linalg.matrix_norm(X0 - X1) / torch.linalg.matrix_norm(X0)) <= 2e-6


CHEBYSHEVS = [(500, 9), (1000, 9), (1450, 4), (1536, 3), (2300, 3)]


def test_these_sizes_reach_every_form(lib):
    """The dispatch sends the sizes above to every form there is, so that what they compare are two forms."""
    got = set()
    for m, n in SIZES:
        plan = lib.Plan(m, n)
        tile, blocks, split = lib.polar_query_form(plan.handle)
        plan.close()
        assert (tile == 0) == (("bf16x6", m, n) in SEPARATE)
        got.add((tile, blocks == 1) + split)
    assert got == {(64, True, 1, 1), (64, False, 4, 4), (64, False, 4, 2), (64, False, 4, 1), (64, False, 2, 2),
                   (64, False, 2, 1), (64, False, 1, 1), (128, False, 1, 1), (0, False, 1, 1)}
    for m, n in SIZES32:
        plan = lib.Plan(m, n, prec="fp32")
        assert lib.polar_query_form(plan.handle)[0] == (0 if ("fp32", m, n) in SEPARATE else 32)
        plan.close()

    def forms(what, sizes):
        return {(f[0],) + f[2] for f in (lib.polar_query_form(None, what, *s) for s in sizes)}

    assert forms(lib.POLAR_FORM_INVERSE, INVERSES + [(300, 300)]) == {(64, 4, 4), (64, 2, 4), (64, 2, 2), (64, 1, 1),
                                                                      (128, 1, 1)}
    assert forms(lib.POLAR_FORM_CHEBYSHEV, [(n, n) for n, _ in CHEBYSHEVS]) == {(64, 4, 1), (64, 2, 1), (64, 1, 1),
                                                                               (128, 1, 1)}
    assert forms(lib.POLAR_FORM_GEMM, [s[:3] for s in GEMMS]) == {(64, 4, 1), (64, 2, 1), (64, 1, 1), (0, 1, 1)}
    # plain products and solves that were measured faster on 128 x 128 tiles, and on 32 x 32 ones
    assert forms(lib.POLAR_FORM_GEMM_FP32, [(448, 5480, 1629), (1279, 887, 115), (2936, 641, 580), (515, 5211, 27),
                                            (718, 2215, 806), (1656, 1757, 478)]) == {(0, 1, 1)}
    assert forms(lib.POLAR_FORM_GEMM_FP32, [(52, 77, 3360), (634, 161, 1509), (4163, 74, 240), (911, 625, 774),
                                            (1883, 539, 3684)] + [s[:3] for s in PLAIN]) == {(32, 1, 1)}
    assert forms(lib.POLAR_FORM_INVERSE, [(4500, 4400)]) == {(0, 1, 1)}
    assert forms(lib.POLAR_FORM_CHEBYSHEV, [(7000, 7000)]) == {(0, 1, 1)}


@pytest.mark.parametrize("n,d", CHEBYSHEVS)
def test_coop_chebyshev_matches_separate_launches(lib, monkeypatch, n, d):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    q, _ = torch.linalg.qr(torch.randn(n, n, device="cuda", dtype=torch.float64, generator=g))
    lam = torch.linspace(-1.0, 1.0, n, device="cuda", dtype=torch.float64)
    a = ((q * lam) @ q.T).float()
    coef = [0.3 / (k + 1.0) for k in range(d + 1)]
    F = torch.empty((n, n), device="cuda")
    lib.polar_chebyshev(a, F, -1.0, 1.0, coef)
    monkeypatch.setenv("POLAR_TC_CTA_PAIR", "0")
    G = torch.empty((n, n), device="cuda")
    lib.polar_chebyshev(a, G, -1.0, 1.0, coef)
    assert torch.equal(F, F.T)
    # d - 1 steps of float32-grade products in either form (2e-6: the bound of the form's own test)
    assert float(torch.linalg.matrix_norm(F - G) / torch.linalg.matrix_norm(G)) <= 2e-6


def test_kept_workspace_is_not_shared_between_threads(lib):
    """Concurrent calls of different sizes on streams of their own, after calls that left a block behind:
    each gets the result it gets alone."""
    import threading

    import torch
    mats = [torch.from_numpy(synth.matrix_with_spectrum(n, n, synth.logspace_spectrum(n, 0.3), n)).cuda()
            for n in (150, 260, 400)]
    want = []
    for a in mats:
        X = torch.empty_like(a)
        lib.polar_ns_inverse(a, X)
        want.append(X)
    torch.cuda.synchronize()
    errs = []

    def work(i):
        s = torch.cuda.Stream()
        for _ in range(4):
            X = torch.empty_like(mats[i])
            s.wait_stream(torch.cuda.default_stream())
            lib.polar_ns_inverse(mats[i], X, stream=s)
            if not torch.equal(X, want[i]):
                errs.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errs


def test_kept_workspace_is_given_back(lib):
    import torch
    a = torch.from_numpy(synth.matrix_with_spectrum(1500, 1500, synth.logspace_spectrum(1500, 0.3), 9)).cuda()
    X, Y = torch.empty_like(a), torch.empty_like(a)
    lib.polar_ns_inverse(a, X)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    lib.polar_release_workspace()
    # planes of A, of X twice and of A X, and C = A^T A
    assert torch.cuda.mem_get_info()[0] - held >= (4 * 3 * 2 + 4) * 1500 * 1500
    lib.polar_release_workspace()                   # nothing is kept now
    lib.polar_ns_inverse(a, Y)
    assert torch.equal(X, Y)


_SLICE_PROBE = """
import hashlib, sys, torch
from paper_2112_09017_gb300 import polar, synth
tune = [{"n_lo": 1, "n_hi": 10 ** 6, "aspect_lo": 0.0, "aspect_hi": 1e9, "tile_n": 0, "slice_stages": int(sys.argv[1])}]
def digest(*ts):
    torch.cuda.synchronize()
    return hashlib.sha256(b"".join(t.cpu().numpy().tobytes() for t in ts)).hexdigest()[:16]
a = torch.from_numpy(synth.matrix_with_spectrum(300, 300, synth.logspace_spectrum(300, 0.1), 1)).cuda()
out = []
U, H, info = polar.Plan(300, 300)(a)
out += [info["launches"] > 1, digest(U, H)]
X = torch.empty_like(a)
polar.polar_ns_inverse(a, X)
out.append(digest(X))
s = a + a.T
polar.polar_chebyshev(s, X, -4.0, 4.0, [1.0, 0.5, 0.25, 0.125, 0.0625])
out.append(digest(X))
for t in (None, tune):
    p = polar.polar_batched_plan_create([300], [300], None, tune=t)
    polar.polar_batched_run(p, [a], [U], [H], 0.0, None, None)
    out.append(digest(U, H))
print(*out)
"""


def _slice_probe(stages, env):
    import os
    import subprocess
    import sys
    e = {k: v for k, v in os.environ.items() if not k.startswith("POLAR_TC_")}
    e.update(env)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _SLICE_PROBE, str(stages)], cwd=root, env=e, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.split()


def test_slice_length_of_the_environment_reaches_every_product(lib):
    """POLAR_TC_SLICE_STAGES: the solve, the inverse and the Chebyshev series leave their one-launch forms, whose slices
    are 64 of K, and a batched plan takes it where no table says otherwise. Read once per process, so in others."""
    multi0, solve0, inv0, cheb0, batch0, tuned0 = _slice_probe(4, {})
    multi4, solve4, inv4, cheb4, batch4, tuned4 = _slice_probe(4, {"POLAR_TC_SLICE_STAGES": "4"})
    assert (multi0, multi4) == ("False", "True")
    assert solve4 != solve0 and inv4 != inv0 and cheb4 != cheb0
    assert batch0 != tuned0 and batch4 == tuned4 == tuned0


@pytest.mark.parametrize("kind", ["solve", "fp32", "batch"])
def test_a_plan_is_ready_for_any_stream(lib, kind):
    """A plan made while the default stream is busy, run at once on a stream that does not wait for it: the clearing
    of the plan's buffers is over when the plan is returned."""
    import torch
    n = 700
    a = torch.from_numpy(synth.matrix_with_spectrum(n, n, synth.logspace_spectrum(n, 0.1), 21)).cuda()
    outs = []
    U, H = torch.empty_like(a), torch.empty_like(a)
    for busy in (False, True):
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(400_000_000)            # about 0.2 s of the default stream
        if kind == "batch":
            plan = lib.polar_batched_plan_create([n], [n])
            lib.polar_batched_run(plan, [a], [U], [H], 0.0, None, None, stream=s)
        else:
            plan = lib.Plan(n, n, prec="bf16x6" if kind == "solve" else "fp32")
            plan(a, U=U, H=H, stream=s)
        torch.cuda.synchronize()
        outs.append((U.clone(), H.clone()))
        if kind == "batch":
            lib.polar_plan_destroy(plan)
        else:
            plan.close()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("kind,m,n,count", [("bf16x6", 400, 300, 4), ("bf16x6", 1000, 700, 3), ("bf16x6", 2100, 2050, 2),
                                            ("fp32", 300, 200, 4), ("batch", 500, 400, 3)], ids=lambda v: str(v))
def test_one_launch_kernels_on_streams_of_their_own(lib, kind, m, n, count):
    """Plans run at the same time from threads, each on its own stream, together more blocks than the GPU holds: a
    cooperative launch starts when all of its blocks fit, so none waits for blocks that cannot start, and each
    returns what it returns alone."""
    import threading

    import torch
    mats = [torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 0.1), 70 + i)).cuda()
            for i in range(count)]
    streams = [torch.cuda.Stream() for _ in range(count)]
    outs = [[(torch.empty_like(a), torch.empty((n, n), device="cuda")) for _ in range(2)] for a in mats]
    if kind == "batch":
        plans = [lib.polar_batched_plan_create([m], [n]) for _ in mats]
    else:
        plans = [lib.Plan(m, n, prec=kind) for _ in mats]
    torch.cuda.synchronize()                 # the inputs are there for every stream

    def run(i, rep):
        U, H = outs[i][rep]
        if kind == "batch":
            lib.polar_batched_run(plans[i], [mats[i]], [U], [H], 0.0, None, None, stream=streams[i])
            streams[i].synchronize()
        else:
            plans[i](mats[i], U=U, H=H, stream=streams[i])

    for i in range(count):
        run(i, 0)
    errs = []

    def work(i):
        try:
            for _ in range(5):
                run(i, 1)
        except Exception as e:               # a timeout's status, for the assertion below
            errs.append(e)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(count)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errs
    for (U, H), (U2, H2) in outs:
        assert torch.equal(U, U2) and torch.equal(H, H2)
    for p in plans:
        lib.polar_plan_destroy(p) if kind == "batch" else p.close()
