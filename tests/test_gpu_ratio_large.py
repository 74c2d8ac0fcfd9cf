"""The class-ratio ranking where a count is too large for the quotients alone
(2^25 and more: the ranking kernel compares exactly), beside entries with equal
quotients, for the list lengths around its 256-entry slices."""
import numpy as np
import pytest

import oracle
from test_gpu_batched import check_ratio, ctr, run_batched  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [3, 255, 256, 300])
def test_ratio_with_a_large_count(ctr, extra):  # noqa: F811
    words = [bytes([97 + i % 26, 97 + i // 26 % 26, 98]) for i in range(extra)]
    docs = [b"a " * ((1 << 25) + 3) + b" ".join(words), b" ".join(words[::2] * 2) + b" a a", b" ".join(words[::3])]
    text = np.frombuffer(b"\n".join(docs), np.uint8)
    offs = np.cumsum([0] + [len(d) + 1 for d in docs]).astype(np.uint64)
    offs[-1] = text.size
    cls = np.array([0, 1, 1], np.uint32)
    r = oracle.count(text, offs, cls, 2)
    b, keep = run_batched(ctr, text, offs, cls, 2, checked=True)
    for c in range(2):
        for k in (1, 50, 64):
            check_ratio(ctr, b, r, c, k)
