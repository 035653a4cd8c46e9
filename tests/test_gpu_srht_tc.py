"""Mixed SRHT passes on the tensor cores (groups of 2^10 and 2^11 rows): every combination of the two,
ragged rows and columns, a row stride, outputs whose rows are not 16-byte aligned, columns of very
different scale, and non-finite values."""
import numpy as np
import pytest

from oracle import sketch as osk
from tests.gpu_helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slse():
    torch_cuda()
    import paper_2509_06856_gb300 as m
    return m


def _compare(SX, ox):
    # two roundings to BF16 (8 significant bits: at most 2^-8 relative each), the first on the
    # intermediate, whose 2^9 to 2^11 rounding errors of an entry add up as independent terms: six
    # standard deviations of 2^-8 / sqrt(3) of the column's root mean square, and 2^-8 of the entry
    rms = np.sqrt((ox ** 2).mean(0)) + 1e-300
    err = np.abs(host(SX) - ox)
    assert np.all(err <= 6 * 2.0 ** -8 / np.sqrt(3.0) * rms + 2.0 ** -8 * np.abs(ox))


# N' = 2^19 (10 + 9), 2^20 (10 + 10), 2^21 (11 + 10), 2^22 (11 + 11)
@pytest.mark.parametrize("N,d,ld", [((1 << 19) - 3, 8, 8), ((1 << 19) + 1, 70, 72), (1 << 20, 33, 36), ((1 << 20) + 77, 5, 8),
                                    ((1 << 21) - 1, 40, 40), ((1 << 21) + 9, 17, 20), ((1 << 22) - 5, 12, 12)])
def test_tensor_core_passes_match_the_oracle(slse, N, d, ld):
    rng = np.random.default_rng(N + d)
    wide = np.zeros((N, ld), np.float32)
    wide[:, :d] = rng.standard_normal((N, d)) * 2.0 ** np.linspace(-40, 40, d)
    wide[:, d:] = np.nan  # beyond the columns: never used
    Y = rng.standard_normal(N).astype(np.float32)
    m = 1 << 15
    SX, _ = slse.sketch(dev(wide)[:, :d], dev(Y), m, seed=3, prec="mixed_bf16")
    ox, _ = osk.sketch(wide[:, :d].astype(np.float64), Y.astype(np.float64), m, 3)
    _compare(SX, ox)


@pytest.mark.parametrize("N,d", [((1 << 19) + 5, 24), ((1 << 21) + 5, 12)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_columns_stay_apart(slse, N, d, bad):
    rng = np.random.default_rng(N)
    X, Y = rng.standard_normal((N, d)).astype(np.float32), rng.standard_normal(N).astype(np.float32)
    X[N // 2, 3] = bad
    SX, _ = slse.sketch(dev(X), dev(Y), 4096, seed=2, prec="mixed_bf16")
    with np.errstate(all="ignore"):
        ox, _ = osk.sketch(X.astype(np.float64), Y.astype(np.float64), 4096, 2)
    got = host(SX)
    assert np.array_equal(np.isnan(got), np.isnan(ox))
    assert np.array_equal(np.isposinf(got), np.isposinf(ox))
    others = [c for c in range(d) if c != 3]
    _compare(SX[:, others], ox[:, others])


def test_fp32_split_is_exact(slse):
    # one row of H is all ones: with m = N' every output row is kept, and the rows of the
    # transform of a single non-zero row are that row times +-1 / sqrt(N') up to BF16 rounding
    N, d = 1 << 19, 16
    X = np.zeros((N, d), np.float32)
    X[12345] = np.float32(1.0) + np.arange(d, dtype=np.float32) * np.float32(2.0 ** -23)
    X[12345, 8:] = np.float32(2.0 ** -120) * (1 + np.arange(8, dtype=np.float32) * np.float32(2.0 ** -23))
    SX, _ = slse.sketch(dev(X), dev(np.zeros(N, np.float32)), 1 << 12, seed=1, prec="mixed_bf16")
    want = np.abs(X[12345].astype(np.float64)) / np.sqrt(1 << 12)
    assert np.all(np.abs(np.abs(host(SX)) - want) <= 2.0 ** -8 * want)
