"""The global table of documents that share no word: its first size, a quarter of
the documents' rows, overflows; the second one expects more rows than the bucket
sort takes (5 M), so the table is radix sorted.  The second build must use nothing of the
first one's scratch.  Against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same
from test_gpu_batched import ctr, run_batched  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("docs,words", [(600, 1000), (5500, 1000)])
def test_overflowing_global_table(ctr, docs, words):  # noqa: F811
    from paper_2206_05269_gb300 import wc
    n = np.random.default_rng(docs).choice(26 ** 5, docs * words, replace=False)
    w = np.full((n.size, 6), ord(" "), np.uint8)
    for j in range(5):
        w[:, j] = 97 + n // 26 ** j % 26
    text = w.reshape(-1)
    offs = (np.arange(docs + 1) * words * 6).astype(np.uint64)
    cls = (np.arange(docs) % 2).astype(np.uint32)
    r = oracle.count(text, offs, cls, 2)
    b, keep = run_batched(ctr, text, offs, cls, 2, checked=True)
    assert_same(b.table(wc.WC_TABLE_GLOBAL).export(), r.glob(), "global")
    for c in range(2):
        assert_same(b.table(wc.WC_TABLE_CLASS, c).export(), r.cls(c), f"class {c}")
    b.free()
