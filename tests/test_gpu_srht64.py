"""FP64 SRHT passes in block fixed point: every group size it serves (2^8 .. 2^12 rows), ragged
rows and columns, both storages, columns of very different scale, and elements far below their
column's largest."""
import numpy as np
import pytest

from oracle import sketch as osk
from tests.gpu_helpers import dev, host, padded, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slse():
    torch_cuda()
    import paper_2509_06856_gb300 as m
    return m


# (rows, columns): pass splits 8+7, 8+8, 9+9, 10+9, 10+10, 11+10, 11+11, 12+11
@pytest.mark.parametrize("N,d", [(20000, 17), (1 << 16, 9), ((1 << 17) + 3, 16), ((1 << 18) + 1, 8), ((1 << 20) - 5, 7),
                                 ((1 << 20) + 7, 5), ((1 << 21) + 1, 3), ((1 << 22) + 9, 2)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_fixed_point_passes_match_the_oracle(slse, N, d, dtype):
    rng = np.random.default_rng(N + d)
    X = rng.standard_normal((N, d)) * 2.0 ** np.linspace(-60, 60, d)          # columns of other scales
    X[rng.integers(0, N, N // 8)] *= 2.0 ** rng.integers(-60, 1, (N // 8, 1))  # rows far below them
    X[rng.integers(0, N, 50), rng.integers(0, d, 50)] = 0.0
    X = X.astype(dtype)
    Y = rng.standard_normal(N).astype(dtype)
    m = N // 3
    SX, _ = slse.sketch(dev(X), dev(Y), m, seed=5, prec="fp64")
    ox, _ = osk.sketch(X.astype(np.float64), Y.astype(np.float64), m, 5)
    # every rounding of either side is at most 2^-53 of a partial sum (at most sum |x| of the
    # column): log2 N' levels and the scale in the oracle, two roundings, the scale and the
    # alignment (2^-82 per element) here
    levels = padded(N).bit_length() + 5
    bound = levels * 2.0 ** -53 * np.abs(X.astype(np.float64)).sum(0) / np.sqrt(m)
    assert np.all(np.abs(host(SX) - ox) <= bound)


@pytest.mark.parametrize("N,d", [(20000, 17), ((1 << 18) + 1, 8), ((1 << 20) + 7, 3)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_columns_stay_apart(slse, N, d, bad):
    # one non-finite element: its own column is non-finite as in the oracle, all others stay as they were
    rng = np.random.default_rng(N)
    X, Y = rng.standard_normal((N, d)), rng.standard_normal(N)
    clean, _ = slse.sketch(dev(X), dev(Y), 4096, seed=2, prec="fp64")
    X[N // 2, 1] = bad
    SX, _ = slse.sketch(dev(X), dev(Y), 4096, seed=2, prec="fp64")
    ox, _ = osk.sketch(X, Y, 4096, 2)
    got = host(SX)
    assert np.array_equal(np.isnan(got), np.isnan(ox))
    assert np.array_equal(np.isposinf(got), np.isposinf(ox))
    others = [c for c in range(d) if c != 1]
    bound = 1e-12 * np.sqrt((X[:, others] ** 2).sum(0) / 4096)
    assert np.all(np.abs(got[:, others] - host(clean)[:, others]) <= bound)


def test_power_of_two_range_limits(slse):
    # elements near both ends of the FP64 range: results that leave the normal range round as FP64 does
    rng = np.random.default_rng(3)
    N = 1 << 16
    for p in (-1060, -1022, 1000):
        X = np.ldexp(rng.standard_normal((N, 4)), p)
        SX, _ = slse.sketch(dev(X), dev(rng.standard_normal(N)), N, seed=4, prec="fp64")
        ox, _ = osk.sketch(X, np.zeros(N), N, 4)
        # one unit of the smallest denormal per rounding on top of the relative bound
        bound = 22 * (2.0 ** -53 * np.abs(X).sum(0) / np.sqrt(N) + 256 * 2.0 ** -1074)
        assert np.all(np.abs(host(SX) - ox) <= bound)
