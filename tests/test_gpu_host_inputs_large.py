"""slse_fit with pinned X at transforms whose first pass is the tensor-core or the fixed-point form: the
pass reads X from host memory and stores the device copy that the 2nd stage reads.  The same bits as
from device memory."""
import numpy as np
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


# N' = 2^19 (groups of 2^10 rows) and 2^21 (2^11); 12 columns: aligned rows with a partial slab, 10: rows
# of the cluster form
@pytest.mark.parametrize("N", [(1 << 18) + 5, (1 << 20) + 5])
@pytest.mark.parametrize("dtype,prec", [("float32", "mixed_bf16"), ("float32", "mixed_fp8"), ("float32", "fp64"),
                                        ("float64", "fp64")])
@pytest.mark.parametrize("d", [10, 12, 64])
def test_pinned_x_gives_the_same_bits(N, dtype, prec, d):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    g = torch.Generator(device="cuda").manual_seed(N + d)
    X = torch.randn(N, d, generator=g, device="cuda", dtype=getattr(torch, dtype))
    X[N // 3, d - 1] = 1e-41 if dtype == "float32" else 1e-310     # a denormal
    Y = X[:, 0] + 0.1 * torch.randn(N, generator=g, device="cuda", dtype=X.dtype)
    Xh, Yh = X.cpu().pin_memory(), Y.cpu().pin_memory()
    sched = slse.default_schedule(N, d, prec=prec, T=30, tol=1e-9)
    ref = slse.fit(X, Y, sched, seed=4)
    res = slse.fit(Xh, Yh, sched, seed=4)
    assert res.status == ref.status and res.report["ms_copy_in"] > 0.0
    assert np.array_equal(res.beta, ref.beta)
    assert torch.equal(Xh, X.cpu())
