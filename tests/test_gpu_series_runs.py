"""The series sums at the lengths where the kernel's method changes: the first
run after the directly computed terms (2^16, 2^17), the first full-length runs
(2^21, 2^22), quartic to cubic (2^24, 2^25) and the cubic's longer runs (2^25 to
2^27), against exact sums in whole numbers."""
import numpy as np
import pytest

from test_gpu_series import ctr, gpu_sum  # noqa: F401

pytestmark = pytest.mark.gpu

NS = sorted({(1 << p) + d for p in (15, 16, 17, 21, 22, 24, 25, 26, 27) for d in (-1, 1, 9)} |
            {65_536 + 7 * 8 + 3, 131_072 + 7 * 8 + 3, 70_000_001, 100_000_000})


@pytest.mark.parametrize("series", [0, 1])
def test_series_where_the_method_changes(ctr, series):  # noqa: F811
    b0, b1 = ((26, 52), (40, 80))[series]  # a term is hi / 2^b0 + lo / 2^b1 with whole hi and lo
    total, at = 0, 0
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
        assert gpu_sum(ctr, series, n) == total / (1 << b1), n
