"""FP64 residual-gradient pass with x.beta in block fixed point: every register tile (columns per
lane, scalar and vector loads), rows and coefficients of very different scale, and the values that
take the FP64 sums instead (denormals, infinities, NaNs, products outside the fixed-point range)."""
import numpy as np
import pytest

from tests.gpu_helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def slse():
    torch_cuda()
    import paper_2509_06856_gb300 as m
    return m


def _check(slse, X, Y, beta):
    # FP64 summation of either side: at most n roundings of 2^-53 of a partial sum, for x.beta (n = d)
    # and for the sum over rows (n = N), on sum |x_ij| (|y_i| + sum_k |x_ik beta_k|)
    g = host(slse.grad(dev(X), dev(Y), beta, prec="fp64"))
    X, Y = X.astype(np.float64), Y.astype(np.float64)
    ref = X.T @ (Y - X @ beta)
    bound = 2 * (X.shape[1] + X.shape[0]) * U * (np.abs(X).T @ (np.abs(Y) + np.abs(X) @ np.abs(beta)))
    assert np.all(np.abs(g - ref) <= bound + 1e-300)


@pytest.mark.parametrize("d", [1, 31, 32, 33, 64, 66, 97, 128, 130, 192, 193, 200, 256, 257, 320, 384, 385, 386, 511, 512])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_tiles_and_scales(slse, d, dtype):
    rng = np.random.default_rng(d)
    N = 1000 + d
    col = 2.0 ** rng.integers(-20, 21, d)
    X = rng.standard_normal((N, d)) * col * 2.0 ** rng.integers(-25, 26, (N, 1))
    X[rng.random((N, d)) < 0.1] = 0.0
    X[N // 3] = 0.0                                         # a zero row
    beta = rng.standard_normal(d) / col * 2.0 ** rng.integers(-10, 11, d)
    beta[rng.integers(0, d)] = 0.0
    _check(slse, X.astype(dtype), rng.standard_normal(N).astype(dtype), beta)


@pytest.mark.parametrize("dtype,lo,hi", [(np.float64, -1060, 900), (np.float32, -140, 120)])
def test_range_limits(slse, dtype, lo, hi):
    rng = np.random.default_rng(7)
    N, d = 300, 70
    for p in (lo, hi, 0):
        X = np.ldexp(rng.standard_normal((N, d)), p).astype(dtype)
        X[5, 3] = np.ldexp(1.0, lo)
        beta = np.ldexp(rng.standard_normal(d), min(-p, 1000))  # finite: 2^1060 is not
        _check(slse, X, rng.standard_normal(N).astype(dtype) * dtype(1e-3), beta)
    _check(slse, rng.standard_normal((N, d)).astype(dtype), rng.standard_normal(N).astype(dtype), np.zeros(d))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_values_propagate(slse, dtype, bad):
    rng = np.random.default_rng(9)
    N, d = 500, 40
    X, Y, beta = rng.standard_normal((N, d)).astype(dtype), rng.standard_normal(N).astype(dtype), rng.standard_normal(d)
    for where in ("x", "y", "beta"):
        Xb, Yb, bb = X.copy(), Y.copy(), beta.copy()
        if where == "x":
            Xb[77, 5] = bad
        elif where == "y":
            Yb[77] = bad
        else:
            bb[5] = bad
        g = host(slse.grad(dev(Xb), dev(Yb), bb, prec="fp64"))
        with np.errstate(all="ignore"):
            ref = Xb.astype(np.float64).T @ (Yb.astype(np.float64) - Xb.astype(np.float64) @ bb)
        assert not np.isfinite(ref).any()
        assert not np.isfinite(g).any()
