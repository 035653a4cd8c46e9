"""QR by panels: fewer columns than a panel, ragged last panels, fewer rows than the cluster, one, two and
four rows per thread, the row count from which the column-by-column form runs, a row stride, and a
zero column."""
import numpy as np
import pytest

from oracle import linalg
from tests.gpu_helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,d,pad", [(3, 2, 0), (7, 7, 0), (17, 9, 3), (33, 16, 0), (300, 50, 0), (700, 163, 5), (4096, 8, 0),
                                     (4113, 12, 0), (8200, 20, 0), (16384, 5, 0), (16385, 5, 0)])
def test_panels_match_the_oracle(r, d, pad):
    torch_cuda()
    import paper_2509_06856_gb300 as slse
    A = np.random.default_rng(r * 7 + d).standard_normal((r, d + pad))
    R, H = slse.qr(dev(A)[:, :d])
    A = A[:, :d]
    s = np.linalg.svd(A, compute_uv=False)
    kappa, n = s[0] / s[-1], r * np.sqrt(d)
    Ro = linalg.householder_r(A)
    # normwise backward error of Householder QR at most about r sqrt(d) u on either side, and the
    # first-order sensitivity of R, sqrt(2) kappa
    assert np.linalg.norm(host(R) - Ro) <= 4 * np.sqrt(2) * kappa * n * 2.0 ** -53 * np.linalg.norm(A)
    assert np.all(np.tril(host(R), -1) == 0.0) and np.all(np.diag(host(R)) >= 0.0)
    Hi = np.linalg.inv(Ro.T @ Ro)
    assert np.linalg.norm(host(H) - Hi) <= 16 * kappa ** 2 * n * 2.0 ** -53 * np.linalg.norm(Hi)


def test_zero_column_raises_enumeric():
    torch_cuda()
    import paper_2509_06856_gb300 as slse
    X = np.random.default_rng(1).standard_normal((4096, 24))
    X[:, 17] = 0.0
    sched = slse.default_schedule(4096, 24, T=20, tol=1e-10)
    res = slse.fit(dev(X), dev(X[:, 0].copy()), sched, seed=2, raise_on_error=False)
    assert res.status == slse.ENUMERIC


def test_fit_with_a_workspace_without_the_panels_scratch():
    """One 256-byte unit less than the full workspace: the factor column by column, the same fit within
    the error of either factor; a workspace short by far more stays refused."""
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    rng = np.random.default_rng(4)
    N, d = 5000, 40
    X = rng.standard_normal((N, d))
    Xd, Yd = dev(X), dev(X @ rng.standard_normal(d) + 0.1 * rng.standard_normal(N))
    sched = slse.default_schedule(N, d, prec="fp64", T=60, tol=1e-13)
    full = slse.workspace_size(Xd, Yd, slse.OP_FIT, sched)
    b = [slse.fit(Xd, Yd, sched, seed=6, workspace=slse.alloc_workspace(n)).beta for n in (full, full - 256)]
    # both stop at the fixed point of the same FP64 iteration (tol 1e-13, condition below 2)
    assert np.linalg.norm(b[0] - b[1]) <= 1e-11 * np.linalg.norm(b[0])
    with pytest.raises(slse.SlseError):
        slse.fit(Xd, Yd, sched, seed=6, workspace=slse.alloc_workspace(full // 2))
