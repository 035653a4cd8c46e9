"""Backward solve in correction form (X of 2^24 elements and more): the same solution as the full form
and as the normal equations, aligned and unaligned rows, and a workspace without room for the Gram
matrix (the full form then)."""
import numpy as np
import pytest

import workloads
from tests.gpu_helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d", [((1 << 18) + 5, 64), (1 << 19, 33), ((1 << 15) + 1, 512)])
def test_correction_form_solves_the_normal_equations(N, d):
    torch_cuda()
    import paper_2509_06856_gb300 as slse
    assert N * d >= 1 << 24
    p = workloads.cfg3(N=N, d=d, seed=d)
    X, Y = dev(p["X"]), dev(p["Y"])
    sched = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=1e-9)
    H = slse.fit(X, Y, sched, seed=1, hinv=True).hinv
    v = np.random.default_rng(2).standard_normal(d)
    X64 = p["X"].astype(np.float64)
    want = np.linalg.solve(X64.T @ X64, v)
    got = {}
    for form in ("correction", "full"):
        sched.stage2 = form
        w, rep = slse.solve_normal(X, H, dev(v), sched)
        got[form] = host(w)
        assert rep["status"] in (slse.OK, slse.ENOTCONV)
    # both forms end at the rounding floor of the FP32 passes (1.3e-8 at 16385 x 512, 1e-9 at 2^18 x 33),
    # where one iterate's error is as likely above the other's as below: within a factor of two
    err = {form: np.linalg.norm(w - want) / np.linalg.norm(want) for form, w in got.items()}
    assert err["correction"] <= 2 * max(err["full"], 1e-9), err
    sched.stage2 = "correction"
    need = slse.solve_normal_workspace(X, sched)
    d8 = d * d * 8
    small = slse.alloc_workspace(need - d8)  # the Gram matrix does not fit any more
    w, _ = slse.solve_normal(X, H, dev(v), sched, workspace=small)
    assert np.array_equal(host(w), got["full"])
