"""The fit's iteration kernels as dependent launches: on both sides of the size from which the
correction form's 1st stage uses plain launches (N d = 2^29), and in the full form, where every
launch is a dependent one.  Against FP64 normal equations of the same data: X well conditioned
(i.i.d. normal), Y = X b + noise, so the mixed path's 1e-8 bound applies to each form."""
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d", [((1 << 21) - 3, 256), (1 << 21, 256), (40001, 24)])
@pytest.mark.parametrize("stage2", ["correction", "full"])
def test_fit_on_both_sides_of_the_rule(N, d, stage2):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    g = torch.Generator(device="cuda").manual_seed(5)
    X = torch.randn((N, d), generator=g, device="cuda")
    Y = X @ torch.randn(d, generator=g, device="cuda") + 0.1 * torch.randn(N, generator=g, device="cuda")
    G = torch.zeros((d, d), dtype=torch.float64, device="cuda")
    c = torch.zeros(d, dtype=torch.float64, device="cuda")
    for i in range(0, N, 1 << 19):
        Xc = X[i:i + (1 << 19)].double()
        G += Xc.T @ Xc
        c += Xc.T @ Y[i:i + (1 << 19)].double()
    ref = torch.linalg.solve(G, c).cpu()
    sched = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=1e-10, stage2=stage2)
    res = slse.fit(X, Y, sched, seed=3)
    err = float((torch.as_tensor(res.beta) - ref).norm() / ref.norm())
    print(f"N={N} d={d} {stage2}: {err:.2e}, iterations {res.report['iters_stage2']}")
    assert err <= 1e-8
    # the device clock's sums cover the passes that ran
    assert res.report["n_grad2"] > 0 and 0.0 < res.report["ms_grad2"] < res.report["ms_total"]
    assert (res.report["n_corr"] > 0) == (stage2 == "correction")
