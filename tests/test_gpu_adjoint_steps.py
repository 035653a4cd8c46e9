"""Backward solve on the mixed path at 2^24 elements of X and more: T steps are T passes over FP32 X,
whatever the schedule's 2nd-stage form, so that a solve which ends by T is as close as T steps of the
iteration get, for ill-conditioned X too."""
import numpy as np
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d", [((1 << 18) + 5, 64), (1 << 19, 33)])
@pytest.mark.parametrize("cond", [1.0, 1e3])
def test_steps_are_passes_over_x(N, d, cond):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    g = torch.Generator(device="cuda").manual_seed(d)
    V, _ = torch.linalg.qr(torch.randn(d, d, generator=g, device="cuda", dtype=torch.float64))
    s = torch.logspace(0.0, -np.log10(cond), d, dtype=torch.float64, device="cuda")
    X = torch.randn(N, d, generator=g, device="cuda") @ (s[:, None] * V.T).float()
    Y = torch.randn(N, generator=g, device="cuda")
    v = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
    G = X.double().T @ X.double()
    L = torch.linalg.cholesky(G)
    want = torch.cholesky_solve(v[:, None], L)[:, 0]
    norm = lambda w: float((L.T @ w).norm())  # noqa: E731  ||X w||
    sched = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=1e-9)
    H = slse.fit(X, Y, sched, seed=1, hinv=True).hinv
    rho = np.sqrt(d / sched.r)
    for T in (8, 20):
        sched.T, sched.tol = T, 0.0
        got = {}
        for form in ("correction", "full"):
            sched.stage2 = form
            got[form], rep = slse.solve_normal(X, H, v, sched)
            assert rep["iters_stage2"] == T
        assert torch.equal(got["correction"], got["full"])
        # the iteration's error after T steps is at most about (T + 1) rho^T of the solution in the
        # norm of X (a double root); ten times that for a sketch off its asymptotic rate.  The passes'
        # own error (1e-8) is far below
        assert norm(got["correction"] - want) <= 10 * (T + 1) * rho ** T * norm(want), T


def test_workspace_holds_no_copy_of_x():
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    N, d = 1 << 20, 64
    X = torch.empty((N, d), device="cuda")
    sched = slse.default_schedule(N, d, prec="mixed_bf16")
    # two vectors of N values in FP32, a d x d matrix, and one partial gradient for each of 2 CTAs per
    # SM (at most 256 SMs) beside a few vectors of d values
    assert slse.solve_normal_workspace(X, sched) <= 8 * N + 8 * d * d + (512 + 64) * d * 8 + (1 << 16)
