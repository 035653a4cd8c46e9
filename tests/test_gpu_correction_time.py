"""report.ms_corr: the time of the correction steps' d x d products, whatever the 2nd stage waits for
before them (the Gram matrix is formed beside its first pass)."""
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def test_time_of_a_product_does_not_depend_on_the_rows():
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    d, per = 127, {}
    for N in (1 << 16, 1 << 22):  # the second one's Gram matrix takes longer than its first pass
        g = torch.Generator(device="cuda").manual_seed(N)
        X = torch.randn(N, d, generator=g, device="cuda")
        Y = 3 * X[:, 0] + 0.1 * torch.randn(N, generator=g, device="cuda")
        sched = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=1e-10, kind="countsketch")
        for _ in range(3):
            r = slse.fit(X, Y, sched, seed=1).report
            assert r["n_corr"] > 0
            per[N] = min(per.get(N, 1e9), r["ms_corr"] / r["n_corr"])
    assert per[1 << 22] <= 2 * per[1 << 16], per
