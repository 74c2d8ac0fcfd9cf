"""Class and global tables of which some are bucket sorted and some, being
larger, radix sorted: right, and the small ones finished together, whatever
their number."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same
from test_gpu_batched import ctr, run_batched  # noqa: F401

pytestmark = pytest.mark.gpu

WORDS = 2_700_000  # of each of two documents of class 0: its table and the global one expect more than 5 M rows


def distinct(seed: int) -> bytes:
    n = np.random.default_rng(seed).choice(26 ** 5, WORDS, replace=False)
    w = np.full((WORDS, 6), ord(" "), np.uint8)
    for j in range(5):
        w[:, j] = 97 + n // 26 ** j % 26
    return w.tobytes()


def test_small_tables_beside_large_ones(ctr):  # noqa: F811
    from paper_2206_05269_gb300 import wc
    rng = np.random.default_rng(0)
    vocab = [bytes(rng.integers(97, 123, 1 + i % 24).astype(np.uint8)) for i in range(3000)]
    small = [b" ".join(vocab[i] for i in rng.integers(0, 3000, 2000)) + b" " for _ in range(12)]
    docs = [distinct(1), distinct(2)] + small
    text = np.frombuffer(b"".join(docs), np.uint8).copy()
    offs = np.cumsum([0] + [len(d) for d in docs]).astype(np.uint64)
    launches = []
    for nclasses in (2, 7):
        cls = np.array([0, 0] + [1 + d % (nclasses - 1) for d in range(len(small))], np.uint32)
        b, keep = run_batched(ctr, text, offs, cls, nclasses, checked=True)
        assert b.status() == wc.WC_OK
        wc.wc_profile_enable(ctr.ctx, True)
        g = b.table(wc.WC_TABLE_GLOBAL)
        launches.append(wc.wc_profile_read(ctr.ctx)[4])
        wc.wc_profile_enable(ctr.ctx, False)
        if nclasses == 7:
            r = oracle.count(text, offs, cls, nclasses)
            assert_same(g.export(), r.glob(), "global")
            for c in range(nclasses):
                assert_same(b.table(wc.WC_TABLE_CLASS, c).export(), r.cls(c), f"class {c}")
        b.free()
    assert launches[0] == launches[1] > 20, launches
