"""A wait of the SRHT's tensor-core passes that gives up: slse_sketch returns at once, so its output says
it (NaN in every entry), and the fit reports ETIMEOUT.  With the limit restored the same calls give what
they gave before."""
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,prec", [((1 << 18) + 5, "mixed_bf16"), ((1 << 20) + 3, "mixed_bf16"), ((1 << 20) + 3, "mixed_fp8")])
def test_a_wait_that_gives_up_is_seen(N, prec):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    d, m = 252 if N < 1 << 19 else 20, 4096  # groups of 2^10 rows: on the tensor cores from there on
    g = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(N, d, generator=g, device="cuda")
    Y = torch.randn(N, generator=g, device="cuda")
    sched = slse.default_schedule(N, d, prec=prec, T=30, tol=1e-6)
    before = slse.sketch(X, Y, m, seed=3, prec=prec)
    beta = slse.fit(X, Y, sched, seed=3).beta
    prev = slse.debug_spin_limit(1)
    try:
        got = slse.sketch(X, Y, m, seed=3, prec=prec)
        res = slse.fit(X, Y, sched, seed=3, raise_on_error=False)
        torch.cuda.synchronize()
    finally:
        slse.debug_spin_limit(prev)
    if prec == "mixed_fp8":
        assert bool((got[0] == 0x7F).all())  # NaN of E4M3
    else:
        assert bool(torch.isnan(got[0]).all())
    assert bool(torch.isnan(got[-1]).all())
    assert res.status == slse.ETIMEOUT, slse.status_string(res.status)
    after = slse.sketch(X, Y, m, seed=3, prec=prec)
    assert all(torch.equal(a, b) for a, b in zip(before, after))
    assert (slse.fit(X, Y, sched, seed=3).beta == beta).all()
