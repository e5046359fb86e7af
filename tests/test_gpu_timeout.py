"""Failure detection on the GPU without a fault: the tensor-core kernel's bounded
waits expire, the kernel returns on its own, the solve reports POLAR_ETIMEOUT and
the CUDA context stays usable.

The expiry is made on purpose by a test hook (POLAR_TEST_WITHHOLD_TMA=1): the
producer warp issues no copies, so the MMA and epilogue warps wait on barriers
nothing will complete. Every such wait is bounded (about one second); on expiry
the kernel raises its abort flag, the other roles leave their loops, MMAs and
copies (none here) drain, TMEM is freed and the kernel returns.
"""
import os
import time

import numpy as np
import pytest

from paper_2112_09017_gb300 import synth

pytestmark = pytest.mark.gpu


def test_bounded_wait_expires_and_context_survives(lib, monkeypatch):
    import torch
    a = torch.from_numpy(synth.matrix_with_spectrum(300, 200, synth.logspace_spectrum(200, 1e-2), 3)).cuda()
    plan = lib.Plan(300, 200, prec="bf16x6")
    monkeypatch.setenv("POLAR_TEST_WITHHOLD_TMA", "1")
    t0 = time.time()
    U, H, info = plan(a, raw_status=True)
    dt = time.time() - t0
    monkeypatch.delenv("POLAR_TEST_WITHHOLD_TMA")
    assert info["status"] == lib.POLAR_ETIMEOUT
    assert dt < 30.0
    # the same plan and context still work
    U, H, info = plan(a)
    assert info["status"] == lib.POLAR_OK
    u = U.double()
    assert torch.linalg.matrix_norm(u.T @ u - torch.eye(200, dtype=torch.float64, device="cuda")).item() < 1e-4
    plan.close()


def test_product_timeouts_reach_the_caller(lib, monkeypatch):
    """The stream-asynchronous products (polar_gemm, polar_syrk, polar_gemm_noalloc) report an
    expired bounded wait through polar_async_status; the next product on the same stream is
    correct and the status is clear again."""
    import torch
    rng = np.random.default_rng(4)
    a = torch.from_numpy(rng.standard_normal((300, 200)).astype(np.float32)).cuda()
    b = torch.from_numpy(rng.standard_normal((200, 260)).astype(np.float32)).cuda()
    exact = a.double() @ b.double()
    gram = a.double().T @ a.double()
    assert lib.polar_async_status() == lib.POLAR_OK
    calls = [
        ("polar_gemm", lambda c: lib.polar_gemm(a, b, c, prec=lib.POLAR_BF16X6), (300, 260), exact),
        ("polar_gemm_noalloc", lambda c: lib.polar_gemm_noalloc(a, b, c, prec=lib.POLAR_BF16X6), (300, 260), exact),
        ("polar_syrk", lambda c: lib.polar_syrk(a, c, prec=lib.POLAR_BF16X6), (200, 200), gram),
    ]
    for name, call, shape, want in calls:
        c = torch.zeros(shape, device="cuda")
        monkeypatch.setenv("POLAR_TEST_WITHHOLD_TMA", "1")
        t0 = time.time()
        call(c)                                   # enqueued: the call itself returns OK
        st = lib.polar_async_status()
        monkeypatch.delenv("POLAR_TEST_WITHHOLD_TMA")
        assert st == lib.POLAR_ETIMEOUT, (name, st)
        assert time.time() - t0 < 30.0
        assert lib.polar_async_status() == lib.POLAR_OK      # read and cleared
        call(c)
        assert lib.polar_async_status() == lib.POLAR_OK, name
        err = (c.double() - want).abs().max().item()
        assert err <= 1e-4 * want.abs().max().item(), (name, err)


# one block, tiles shared by four blocks, whole tiles 64 and 128 wide; the plain form, whose first block stays away
# from the grid barrier
ONE_LAUNCH = [("fp32", 300, 200),
              ("solve", 96, 64), ("solve", 512, 512), ("solve", 1744, 1312), ("solve", 2304, 2304),
              ("inverse", 300, 300), ("inverse", 1001, 1001), ("inverse", 2300, 2300),
              ("chebyshev", 300, 300), ("chebyshev", 1450, 1450), ("chebyshev", 2300, 2300)]


@pytest.mark.parametrize("kind,m,n", ONE_LAUNCH, ids=lambda v: str(v))
def test_one_launch_forms_expire_and_the_next_call_is_correct(lib, monkeypatch, kind, m, n):
    """The blocks of a one-launch kernel leave at different times, each after its own wait; the last one out clears
    the grid barrier, and the buffers (a plan's, or the block kept between calls) serve the next call."""
    import torch
    a = synth.matrix_with_spectrum_on_device(m, n, synth.logspace_spectrum(n, 0.2), 5, "cuda", torch.float32)
    if kind == "chebyshev":
        a = 0.5 * (a + a.T)
    plan = lib.Plan(m, n, prec="fp32" if kind == "fp32" else "bf16x6") if kind in ("solve", "fp32") else None

    def call():
        if plan:
            U, H, info = plan(a, raw_status=True)
            return info["status"], torch.cat([U, H])
        X = torch.zeros((n, m), device="cuda")
        if kind == "inverse":
            return lib.polar_ns_inverse(a, X, raw_status=True)["status"], X
        return lib.polar_chebyshev(a, X, -1.0, 1.0, [0.3, 1.0, 0.2, 0.1], raw_status=True), X

    status, want = call()
    assert status == lib.POLAR_OK
    monkeypatch.setenv("POLAR_TEST_WITHHOLD_TMA", "1")
    t0 = time.time()
    status, _ = call()
    monkeypatch.delenv("POLAR_TEST_WITHHOLD_TMA")
    assert status == lib.POLAR_ETIMEOUT and time.time() - t0 < 30.0
    status, got = call()
    assert status == lib.POLAR_OK and torch.equal(got, want)
    if plan:
        plan.close()


def test_batched_loop_expires_and_the_next_run_starts_afresh(lib, monkeypatch):
    """A batched plan built while copies are withheld keeps withholding them: each of its runs reports a timeout for
    every problem and leaves U alone, the second as the first (the barrier and the counts are clear again); a plan
    built afterwards solves."""
    import torch
    sizes = [(300, 300), (520, 260), (96, 96), (1000, 700)]
    As = [torch.from_numpy(synth.matrix_with_spectrum(m, n, synth.logspace_spectrum(n, 1e-2), 60 + i)).cuda()
          for i, (m, n) in enumerate(sizes)]
    ms, ns = [m for m, _ in sizes], [n for _, n in sizes]
    it = torch.zeros(len(sizes), dtype=torch.int32, device="cuda")
    monkeypatch.setenv("POLAR_TEST_WITHHOLD_TMA", "1")
    plan = lib.polar_batched_plan_create(ms, ns)
    monkeypatch.delenv("POLAR_TEST_WITHHOLD_TMA")
    for rep in range(2):
        Us = [torch.full_like(a, 7.0) for a in As]
        Hs = [torch.full((n, n), 7.0, device="cuda") for n in ns]
        t0 = time.time()
        lib.polar_batched_run(plan, As, Us, Hs, 0.0, it, None)
        torch.cuda.synchronize()
        assert time.time() - t0 < 30.0
        assert bool((it == torch.iinfo(torch.int32).min).all()), it
        assert all(bool((u == 7.0).all()) for u in Us)
    lib.polar_plan_destroy(plan)
    plan = lib.polar_batched_plan_create(ms, ns)
    lib.polar_batched_run(plan, As, Us, Hs, 0.0, it, None)
    torch.cuda.synchronize()
    lib.polar_plan_destroy(plan)
    assert bool((it >= 0).all()), it
    for u in Us:
        g = u.double().T @ u.double()
        assert float(torch.linalg.matrix_norm(g - torch.eye(len(g), dtype=torch.float64, device="cuda"))) < 1e-4
