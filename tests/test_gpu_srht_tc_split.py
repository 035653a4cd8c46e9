"""Pass 1 of the mixed SRHT on the tensor cores splits each FP32 value into three BF16 terms.  Two rows
that nearly cancel in half of the outputs show each term: their difference is in the second or the
third terms alone."""
import numpy as np
import pytest

from tests.gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


# N' = 2^19 and 2^20: groups of 2^10 rows in pass 1, 2^21 and 2^22: of 2^11
@pytest.mark.parametrize("N,d", [(1 << 19, 8), (1 << 20, 40), (1 << 21, 12), (1 << 22, 8)])
@pytest.mark.parametrize("bits", [6, 12, 20])
def test_difference_of_two_rows(N, d, bits):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    seed, m = 7, 1 << 12
    P, _, _ = slse.draws(N, seed)
    first = 3 * (N >> 3)                       # positions that share their upper bits share a group
    i, j = int(P[first + 5]), int(P[first + 403])
    rng = np.random.default_rng(bits)
    a = (1.0 + rng.random(d)).astype(np.float32)                   # 24 significant bits each
    b = (a * np.float32(1.0 - 2.0 ** -bits)).astype(np.float32)
    X = torch.zeros((N, d), device="cuda")
    X[i] = torch.from_numpy(a).cuda()
    X[j] = torch.from_numpy(b).cuda()
    SX, _ = slse.sketch(X, torch.zeros(N, device="cuda"), m, seed=seed, prec="mixed_bf16")
    got = SX.double().abs().cpu().numpy() * np.sqrt(m)              # a power of two: exact
    # every output is +-(a - b) or +-(a + b), rounded to BF16 once (all other groups are zero, so the
    # second transform copies it): 2^-8 relative.  Without the third terms a - b is off by up to 2^-16,
    # without the second by up to 2^-8: more than that of 2^-20 and 2^-12.
    small, large = np.abs(a.astype(np.float64) - b), a.astype(np.float64) + b
    is_small = got < 0.5 * large
    want = np.where(is_small, small, large)
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * want)
    # each of the two in about half of the sampled rows (4096 of them: five standard deviations)
    assert np.all(np.abs(is_small.mean(0) - 0.5) <= 5 * 0.5 / np.sqrt(m))
