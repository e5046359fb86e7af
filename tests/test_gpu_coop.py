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


def _solve(lib, a, **kw):
    import torch
    m, n = a.shape
    plan = lib.Plan(m, n, prec="bf16x6", **kw)
    U, H, info = plan(torch.from_numpy(a).cuda(), raw_status=True)
    plan.close()
    return to_np(U), to_np(H), info


# one tile, tile edges in rows (128) and columns (64 and 128), an odd and an even number of 64-wide columns
# (the triangle's pairs), k-block remainders, tall and narrow, more tiles than SMs (the 128-wide tiles), the
# largest sizes below the separate launches and the smallest above
SIZES = [(1, 1), (32, 31), (64, 64), (128, 65), (129, 128), (130, 129), (192, 192), (257, 200), (384, 320),
         (2500, 33), (1000, 996), (1300, 1290), (2100, 2050), (2400, 2304)]


@pytest.mark.parametrize("m,n", SIZES, ids=lambda v: str(v))
def test_coop_solve_matches_oracle_and_separate_launches(lib, m, n):
    kappa = 50.0
    a = synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 1.0 / kappa), 40 + n)
    U, H, info = _solve(lib, a)
    # a residual history that may not hold every step sends a plan to the separate launches
    U2, H2, info2 = _solve(lib, a, max_iter=lib.POLAR_HIST + 10)
    assert info["status"] == info2["status"] == lib.POLAR_OK
    assert info["iters"] == info2["iters"]
    assert info["launches"] == 1 or info["launches"] == info2["launches"]
    # the residuals differ by the rounding of G: about 1e-6 of them far from convergence
    for g, w in zip(info["res_hist"], info2["res_hist"]):
        if w > 1e-3:
            assert abs(g - w) <= 1e-4 * w
    assert info["sym_err"] <= 1e-5 and abs(info["normA_F"] - info2["normA_F"]) <= 1e-12 * info["normA_F"]
    # each is within the forward bound 1e-7 kappa of the exact factor
    assert np.linalg.norm(U.astype(np.float64) - U2) / math.sqrt(n) <= 2e-7 * kappa
    ref = ns_polar(a, tol=1e-12, count_tol=1e-6) if n <= 1300 else None
    met = metrics(a, U, H, ref["U"] if ref else None)
    assert met["orth"] <= 5e-6 and met["bwd"] <= 5e-6 and met["hsym"] == 0.0, met
    if ref:
        assert abs(info["iters"] - ref["iters_at"]) <= 1
        assert met["fwd"] <= 1e-7 * kappa, met


def test_coop_statuses_and_reuse(lib):
    """Zero and non-finite input leave U and H untouched, max_iter returns the last iterate, and the same
    plan solves again afterwards, bit for bit the same twice."""
    import torch
    m, n = 300, 260
    a = torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 1e-2), 3)).cuda()
    plan = lib.Plan(m, n, prec="bf16x6", max_iter=20)
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
    plan = lib.Plan(m, n, prec="bf16x6", max_iter=5)
    U3, H3, i3 = plan(a, raw_status=True)
    plan.close()
    assert i3["status"] == lib.POLAR_NOT_CONVERGED and i3["iters"] == 5 and len(i3["res_hist"]) == 6
    assert i3["res_hist"] == i1["res_hist"][:6]
    assert bool(torch.isfinite(U3).all()) and bool(torch.isfinite(H3).all())
