"""Whole documents that hold words of 17+ letters, in every size class: the
block lists its long words behind the short ones while its other warps still
turn the short ones into sort keys, so no word of such a document may take the
longer list's length for the shorter one's.  Against the oracle, row by row."""
import numpy as np
import pytest

import oracle
from test_gpu_batched import check_docs, ctr, run_batched  # noqa: F401

pytestmark = pytest.mark.gpu


def document(rng, size: int, nlong: int) -> bytes:
    """About `size` bytes: words of 1 to 9 letters with unequal counts, and
    nlong different words of 17 to 40 letters (some of one prefix) among them."""
    vocab = [bytes(rng.integers(97, 123, int(n)).astype(np.uint8)) for n in rng.integers(1, 10, 40 + size // 40)]
    words = [vocab[i] for i in (rng.zipf(1.3, size // 7) - 1) % len(vocab)]
    for i in range(nlong):
        w = b"commonprefixofall"[:17 if i % 3 else 9] + bytes(rng.integers(97, 123, 8 + i % 16).astype(np.uint8))
        for at in rng.integers(0, len(words), 1 + i % 3):
            words.insert(int(at), w)
    return b" ".join(words)


@pytest.mark.parametrize("size", [300, 3_000, 12_000, 50_000])
def test_documents_with_long_words(ctr, size):  # noqa: F811
    rng = np.random.default_rng(size)
    docs = [document(rng, size, d % 61) for d in range(min(1500, 6_000_000 // size))]
    text = np.frombuffer(b"\n".join(docs) + b"\n", np.uint8).copy()
    offs = np.cumsum([0] + [len(d) + 1 for d in docs]).astype(np.uint64)
    r = oracle.count(text, offs)
    for _ in range(3):
        b, keep = run_batched(ctr, text, offs, checked=True)
        check_docs(b, r, len(docs))
        b.free()
