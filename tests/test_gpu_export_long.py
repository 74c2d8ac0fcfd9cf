"""Exports of tables of at most 4,096 rows around the limits up to which one
block writes them (16 KB of letters, 24 a row), with words written by a thread
and by a warp: against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu

# rows, letters of most words, letters of three more
CASES = [(1, 5, ()), (1, 24, ()), (1, 25, ()), (100, 24, ()), (100, 25, ()), (682, 24, ()), (683, 24, ()),
         (700, 4, (64, 65, 9_000)), (1500, 4, (64, 65, 9_000)), (30, 2_000, (63, 66, 20_000)), (4093, 3, (64, 65, 1_200)),
         (4096, 4, ()), (4096, 7, ()), (4097, 3, ())]


@pytest.mark.parametrize("rows,letters,more", CASES)
def test_export(rows, letters, more):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    rng = np.random.default_rng(rows + letters)
    words = set()
    while len(words) < rows:
        words.add(bytes(rng.integers(97, 123, letters).astype(np.uint8)))
    words |= {b"c" * k for k in more}
    text = b" ".join(sorted(words))
    ctr = wc.Counter(0)
    table = ctr.count_checked(to_dev(text), opts=(1 << 14, 1 << 14, 2 * len(text) + 65536))
    want = oracle.count(text).glob()
    assert_same(table.export(), want, f"{rows} rows")
    top = ctr.topk(table, 3)
    assert top.as_list() == want.as_list()[:3]
    ctr.close()
