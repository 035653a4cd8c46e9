"""Mixed SRHT pass 1 on both sides of the widths from which it runs on the tensor cores, last slabs of every
fill (units of eight columns, parts of one), aligned and unaligned rows of the output."""
import numpy as np
import pytest

from oracle import sketch as osk
from tests.gpu_helpers import host, torch_cuda

pytestmark = pytest.mark.gpu


# N' = 2^19: from four slabs of 64 columns on; 2^20: where the last slab is more than half full; 2^21: groups of
# 2^11 rows, slabs of 32 columns
@pytest.mark.parametrize("N,widths", [((1 << 19) - 1, (64, 192, 193, 196, 232, 250, 256)),
                                      ((1 << 20) - 3, (32, 33, 36, 37, 40, 61, 96, 100, 121)),
                                      ((1 << 21) - 7, (1, 3, 7, 12, 20, 31, 37, 60))])
def test_widths_match_the_oracle(N, widths):
    torch = torch_cuda()
    import paper_2509_06856_gb300 as slse
    m, seed = 1 << 13, 11
    g = torch.Generator(device="cuda").manual_seed(N)
    full = torch.randn(N, max(widths), generator=g, device="cuda")
    Y = torch.randn(N, generator=g, device="cuda")
    # a column's sketch does not depend on the others: the oracle once, for the columns looked at
    cols = sorted({c for d in widths for c in (0, d // 2, d - 1, max(0, d - 9))})
    ox, oy = osk.sketch(full[:, cols].double().cpu().numpy(), Y.double().cpu().numpy(), m, seed)
    for d in widths:
        ld = (d + 3) // 4 * 4  # rows that the tensor-core form takes
        X = torch.full((N, ld), float("nan"), device="cuda")
        X[:, :d] = full[:, :d]
        SX, SY = slse.sketch(X[:, :d], Y, m, seed=seed, prec="mixed_bf16")
        keep = [k for k, c in enumerate(cols) if c < d]
        got, want = host(SX)[:, [cols[k] for k in keep]], ox[:, keep]
        # two roundings to BF16, the first on the intermediate, whose 2^9 to 2^11 errors of an entry add up as
        # independent terms: six standard deviations of 2^-8 / sqrt(3) of the column's root mean square
        rms = np.sqrt((want ** 2).mean(0))
        assert np.all(np.abs(got - want) <= 6 * 2.0 ** -8 / np.sqrt(3.0) * rms + 2.0 ** -8 * np.abs(want)), d
        assert bool(torch.isfinite(SX.float()).all()), d
