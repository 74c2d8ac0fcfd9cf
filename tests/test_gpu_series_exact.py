"""wc_series_sum is the double nearest to the exact sum of the correctly
rounded terms: compared bit for bit with that sum in whole numbers.

A term is hi / 2^b0 + lo / 2^b1 with whole hi and lo (powers of two, so every
step below is exact), and a ratio of Python ints is rounded to nearest.  The
lengths lie around the kernel's changes of method: the last directly computed
term (2^18, 2^19), the shortest runs, the powers of two that cut runs, and the
long runs (from 2^24 and 2^25)."""
import numpy as np
import pytest

from test_gpu_series import ctr, gpu_sum  # noqa: F401

pytestmark = pytest.mark.gpu

POWERS = [5, 18, 19, 20, 21, 22, 23, 24, 25]
NS = sorted({(1 << p) + d for p in POWERS for d in (-1, 0, 1, 2)} | {4, 7, 1025, 262_147, 300_001, 786_433, 1_500_007,
                                                                    16_777_471, 33_554_691, 35_000_003})


def prefix_sums(series):
    """Exact sums at every length of NS, as Python ints over 2^b1."""
    b0, b1 = ((26, 52), (40, 80))[series]
    total, at, out = 0, 0, {}
    for n in NS:
        while at < n:
            end = min(n, at + (1 << 20))
            i = np.arange(at + 1, end + 1, dtype=np.float64)
            t = np.sqrt(i) if series == 0 else 1.0 / i
            h = np.floor(t * 2.0 ** b0)
            d = (t - h * 2.0 ** -b0) * 2.0 ** b1
            sign = np.where(i % 2 == 1, 1, -1) if series else 1
            total += (int((h.astype(np.int64) * sign).sum()) << (b1 - b0)) + int((d.astype(np.int64) * sign).sum())
            at = end
        out[n] = total / (1 << b1)
    return out


@pytest.mark.parametrize("series", [0, 1])
def test_series_is_the_exactly_rounded_sum(ctr, series):  # noqa: F811
    want = prefix_sums(series)
    got = {n: gpu_sum(ctr, series, n) for n in NS}
    assert got == want
