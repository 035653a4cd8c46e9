"""FP64 residual-gradient pass where x . beta has no non-zero term (beta = 0, rows of zeros): the gradient,
and the time of a pass over ordinary rows."""
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("d", [37, 256, 512])
def test_zero_terms(d, dtype):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    N = (1 << 19) + 3
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(N, d, generator=g, device="cuda", dtype=getattr(torch, dtype))
    Y = torch.randn(N, generator=g, device="cuda", dtype=X.dtype)
    b = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
    ws = slse.alloc_workspace(slse.workspace_size(X, Y, slse.OP_GRAD))

    def best(X, b):
        t = []
        for _ in range(12):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            slse.grad(X, Y, b, prec="fp64", workspace=ws)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        return min(t)

    ordinary = best(X, b)
    half, some = X.clone(), X.clone()
    half[torch.rand(N, generator=g, device="cuda") < 0.5] = 0
    some[torch.rand(N, generator=g, device="cuda") < 0.01] = 0
    left = b.clone()
    left[: d // 2] = 0                     # rows with non-zero terms in half of their columns only
    part = X.clone()
    part[::7, d // 2:] = 0                 # and rows whose non-zero x meet zero beta
    for name, x, v in (("beta = 0", X, torch.zeros_like(b)), ("half the rows zero", half, b),
                       ("1 % of the rows zero", some, b), ("disjoint", part, left)):
        got = slse.grad(x, Y, v, prec="fp64", workspace=ws)
        want = x.double().T @ (Y.double() - x.double() @ v)
        # FP64 summation of either side: sqrt(N) times the rounding of about sqrt(N) terms of |b| + 1
        tol = 64 * 2.0 ** -53 * N * (1 + float(v.norm()))
        assert float((got - want).abs().max()) <= tol, name
        t = best(x, v)
        assert t <= 1.25 * ordinary, f"{name}: {t:.3f} ms against {ordinary:.3f} ms"
