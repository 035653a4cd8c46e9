"""FP64 residual-gradient pass near the solution, many rows: the roundings of x . beta are independent
from row to row, so that the error of the gradient grows as the square root of the rows.  Against a
sum in double-double arithmetic."""
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def _two_prod(a, b):
    """Product and its error by Dekker's splitting."""
    p = a * b
    def split(x):
        c = 134217729.0 * x
        h = c - (c - x)
        return h, x - h
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _gradient(torch, X, Y, beta):
    """X^T (Y - X beta) as an unevaluated sum of two doubles."""
    hi, lo = Y.clone(), torch.zeros_like(Y)
    for j in range(X.shape[1]):
        p, e = _two_prod(X[:, j].contiguous(), -beta[j])
        hi, t = _two_sum(hi, p)
        lo = lo + (t + e)
    hi, lo = _two_sum(hi, lo)
    P, E = _two_prod(X, hi[:, None].expand_as(X))
    E = E + X * lo[:, None]
    while P.shape[0] > 1:
        h = P.shape[0] // 2  # the rows are a power of two
        P, t = _two_sum(P[:h], P[h:])
        E = E[:h] + E[h:] + t
    return P[0], E[0]


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("d", [10, 37])
def test_error_grows_as_the_root_of_the_rows(d, dtype):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    N = 1 << 20
    g = torch.Generator(device="cuda").manual_seed(d)
    dt = getattr(torch, dtype)
    X = torch.randn(N, d, generator=g, device="cuda", dtype=dt)
    b = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
    Y = (X.double() @ b + 1e-3 * torch.randn(N, generator=g, device="cuda", dtype=torch.float64)).to(dt)
    got = slse.grad(X, Y, b, prec="fp64")
    hi, lo = _gradient(torch, X.double(), Y.double(), b)
    err = float(((got - hi) - lo).norm())
    # x . beta (about |b|) rounded once: at most 2^-53 |b|, 0.4 of it as a standard deviation, times
    # an entry of X (1), summed over N rows; the sums of the small residuals round far below
    assert err <= (N * d) ** 0.5 * 2.0 ** -53 * float(b.norm())
