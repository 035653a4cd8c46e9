"""report.kernels of a fit: the kernel launches that the profiler sees."""
import numpy as np
import pytest

import workloads
from tests.gpu_helpers import dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,prec,kind", [(20000, 50, "fp64", "srht"), (20000, 7, "fp64", "srht"), (30000, 163, "fp64", "srht"),
                                           (20000, 40, "fp64", "gaussian"), (40000, 48, "mixed_bf16", "srht"),
                                           (40000, 47, "mixed_bf16", "gaussian"), (400, 8, "mixed_bf16", "srht"),
                                           (40000, 48, "mixed_bf16", "countsketch"), (40000, 31, "fp64", "countsketch")])
def test_kernels_are_the_launches(N, d, prec, kind):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    from torch.profiler import ProfilerActivity, profile
    p = workloads.gaussian(N, d, seed=d)
    X, Y = p["X"], p["Y"]
    if prec != "fp64":
        X, Y = X.astype(np.float32), Y.astype(np.float32)
    X, Y = dev(X), dev(Y)
    sched = slse.default_schedule(N, d, prec=prec, T=40, tol=0.0, kind=kind)
    slse.fit(X, Y, sched, seed=1)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]):  # a process' first one may see nothing
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        res = slse.fit(X, Y, sched, seed=1)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if str(e.device_type).endswith("CUDA")]
    seen = [n for n in names if not n.startswith(("Memset", "Memcpy"))]
    if not seen:
        pytest.skip("the profiler sees no kernels on this machine")
    assert res.report["kernels"] == len(seen)
