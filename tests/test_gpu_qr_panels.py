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


def test_qr_with_a_workspace_without_the_panels_copy():
    """One 256-byte unit less than the full workspace: the factor column by column, R within the error of
    either factor (above); a workspace short by far more stays refused."""
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    r, d = 700, 40
    A = np.random.default_rng(4).standard_normal((r, d))
    Ad = dev(A)
    full = slse.workspace_size(Ad, Ad[:, 0].contiguous(), slse.OP_QR, arg=r)
    got = []
    for n in (full, full - 256, r * d * 4):
        ws = slse.alloc_workspace(n)
        R = torch.zeros((d, d), dtype=torch.float64, device="cuda")
        st = slse._lib.slse_qr(Ad.data_ptr(), r, d, d, R.data_ptr(), None, ws.data_ptr(), n, slse._stream(None))
        torch.cuda.synchronize()
        got.append((st, host(R)))
    assert [g[0] for g in got] == [slse.OK, slse.OK, slse.ENOMEM]
    s = np.linalg.svd(A, compute_uv=False)
    tol = 4 * np.sqrt(2) * s[0] / s[-1] * r * np.sqrt(d) * 2.0 ** -53 * np.linalg.norm(A)
    assert np.linalg.norm(got[0][1] - got[1][1]) <= tol
