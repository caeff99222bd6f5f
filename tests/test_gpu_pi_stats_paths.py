"""The median select on both sides of the one-launch limit (segments of up to 53,248 factors are
selected in one block's shared memory, longer ones by passes over the grid), with the rows
that make a pass special: runs of zeros at the middle, one value, two values, both zeros,
infinities, NaNs and subnormals.  Medians are exact, so the comparison is equality."""
import numpy as np
import pytest
import torch

from paper_1805_08469_gb300 import gem

from test_gpu_pi_stats import _check_medians, _setup  # noqa: F401  (_setup is the module's fixture)

pytestmark = pytest.mark.gpu

LIMIT = 53248


def _rows(rng, P):
    rows = rng.exponential(size=(11, P)).astype(np.float32)
    rows[0] = 0.0
    rows[1, rng.random(P) < 0.5] = 0.0                   # the run of zeros ends near the middle
    rows[2] = -rows[2]
    rows[3] = np.where(rng.random(P) < 0.5, np.float32(-0.0), np.float32(0.0))
    rows[4, rng.random(P) < 0.4] = np.inf
    rows[5] = np.float32(1.5)
    rows[6] = np.where(np.arange(P) % 2 == 0, np.float32(1.0), np.nextafter(np.float32(1.0), np.float32(2.0)))
    rows[7] = (rng.standard_normal(P) * 1e-40).astype(np.float32)
    rows[8, : P // 2] = 0.0                              # lower and upper middle on both sides of the run's end
    rows[8, P // 2:] += 1.0
    rows[9] = np.arange(P, dtype=np.float32)
    rows[10] = (1.0 + rng.integers(0, 2000, P) * 2.0 ** -20).astype(np.float32)   # one first-pass digit
    return rows


@pytest.mark.parametrize("P", [1, 2, 3, 31, 33, 1023, 1025, 16384, 40961, LIMIT - 1, LIMIT, LIMIT + 1, 120_001])
def test_medians_on_both_sides_of_the_limit(P):
    _check_medians(_rows(np.random.default_rng(P), P), [0, P])


@pytest.mark.parametrize("longest", [LIMIT, LIMIT + 1])
def test_segments_up_to_and_past_the_limit(longest):
    """Empty, unit, odd and even segments next to the longest, none aligned."""
    P = longest + 2111
    _check_medians(_rows(np.random.default_rng(longest), P), [1, 1, 2, 4, 7, 7 + longest, 7 + longest, P - 1000, P - 3])


@pytest.mark.parametrize("P", [101, LIMIT + 2])
def test_nan_rows(P):
    """NaNs order above +inf (sign bit clear) or below everything."""
    x = np.linspace(-1, 1, P).astype(np.float32)
    x[: P // 4] = np.nan
    x[P // 4: P // 2] = np.copysign(np.float32(np.nan), np.float32(-1))
    key = x.view(np.int32).astype(np.int64)
    order = np.sort(np.where(key < 0, (-1 - (key & 0xffffffff)) % (1 << 32) - (1 << 32), key))
    lo = torch.empty((1, 1), device="cuda")
    hi = torch.empty((1, 1), device="cuda")
    with gem.Gem(P, 1, 0.01, 0.9, 1e-8) as G:
        G.pi_median([torch.from_numpy(x).cuda()], [0, P], lo, hi)
        G.sync()
    for got, r in ((lo, (P - 1) // 2), (hi, P // 2)):
        k = int(order[r])
        bits = k if k >= 0 else (~k & 0xffffffff) | 0
        want = np.array([bits if k >= 0 else ((-1 - k) % (1 << 32))], dtype=np.uint64).astype(np.uint32)
        assert got.cpu().numpy().view(np.uint32)[0, 0] == want[0]
