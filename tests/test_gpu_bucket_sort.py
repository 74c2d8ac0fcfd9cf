"""The bucket sort of finished tables, (document, word) rows and vocabularies
at the sizes and key distributions where it can go wrong, against the oracle:
no entry to several buckets, entries that differ only in their last letters or
in their counts, runs of words of 17+ letters that tie on count and prefix.
(Buckets sorted in global memory and spilled entries: the one-slot build of
test_gpu_collisions.py, where nearly every bucket is.)  Whole numbers and
bytes: equal."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    c = wc.Counter(0)
    yield c
    c.close()


def letters(i: int, width: int) -> bytes:
    out = bytearray(width)
    for j in range(width - 1, -1, -1):
        out[j] = 97 + i % 26
        i //= 26
    return bytes(out)


def words(kind: str, n: int) -> list[bytes]:
    """n distinct words (each repeated as its kind says), shuffled."""
    rng = np.random.default_rng(n)
    if kind == "random":  # 3 to 16 letters, count 1
        w = {letters(int(rng.integers(0, 26 ** 10)), int(rng.integers(3, 17))) for _ in range(2 * n)}
        w = sorted(w)[:n]
    elif kind == "last":  # one prefix of 11 letters, the last five count up
        w = [b"commonstart" + letters(i, 5) for i in range(n)]
    elif kind == "counts":  # counts from 1 to thousands, few words each
        w = [letters(i, 4) for i in range(n) for _ in range(1 + int(4000 / (1 + i)) + i % 3)]
    else:  # "ties": words of 17 to 21 letters behind one 16-letter word, all counted once
        w = [b"sixteenlettersxx"] + [b"sixteenlettersxx" + letters(i, 1 + i % 5) for i in range(n)]
        w = sorted(set(w))
    rng.shuffle(w)
    return w


CASES = [("random", n) for n in (1, 2, 31, 33, 97, 384, 1500, 20_000, 150_000)] + \
        [("last", n) for n in (5, 500, 3_000, 60_000)] + [("counts", n) for n in (40, 3_000, 12_000)] + \
        [("ties", n) for n in (2, 40, 700)]


@pytest.mark.parametrize("kind,n", CASES)
def test_table_rows_and_vocabulary(ctr, kind, n):
    import torch

    from paper_2206_05269_gb300 import wc
    text = b" ".join(words(kind, n))
    want = oracle.count(text).glob()
    assert_same(ctr.count_checked(to_dev(text, n % 16)).export(), want, "table")
    # the same as two documents: one long enough to be split (its rows sorted
    # behind the document number), one short
    pad = b" qq" * 30_000  # past 64 KB
    docs = [text + pad, b"zz " + text[:2_000]]
    offs = np.array([0, len(docs[0]), len(docs[0]) + len(docs[1])], np.uint64)
    t = to_dev(b"".join(docs))
    b = ctr.count_batched_checked(t, torch.from_numpy(offs.view(np.int64)).cuda(), offs)
    lists = b.doc_lists()
    for d, doc in enumerate(docs):
        assert lists[d] == oracle.count(doc).glob().as_list(), f"document {d}"
    total = oracle.count(docs[0] + b" " + docs[1]).glob()
    assert_same(b.table(wc.WC_TABLE_GLOBAL).export(), total, "global table")
    assert b.vocab().as_list() == sorted(total.as_list()), "vocabulary"
    b.free()
