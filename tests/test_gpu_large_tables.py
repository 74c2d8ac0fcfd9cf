"""Tables on both sides of the sizes up to which the bucket sort finishes them
(10 M slots; for documents split into ranges 5 M expected rows; larger ones are
radix sorted): single and merged tables and split documents, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev
from test_gpu_batched import check_docs, run_batched

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    c = wc.Counter(0, count_bits=32)
    yield c
    c.close()


def text(n: int, seed: int) -> bytes:
    """n words of 1 to 20 letters, many of them different, some of one 16-letter prefix."""
    rng = np.random.default_rng(seed)
    vocab = [bytes(rng.integers(97, 123, 1 + i % 12).astype(np.uint8)) for i in range(n // 2)]
    vocab += [b"sixteenlettersxx" + bytes(rng.integers(97, 100, i % 5).astype(np.uint8)) for i in range(100)]
    pick = np.concatenate([rng.integers(0, len(vocab), n), (rng.zipf(1.3, n) - 1) % len(vocab)])
    return b" ".join([vocab[i] for i in pick])


@pytest.mark.parametrize("slots", [1 << 22, 1 << 23])
def test_single_and_merged_tables(ctr, slots):
    opts = (slots, 4096, 1 << 20)
    a, b = text(60_000, 1), text(60_000, 2)
    ta, tb = ctr.count(to_dev(a), opts=opts), ctr.count(to_dev(b), opts=opts)
    merged = ctr.merge([ta, tb])  # sized by the tables' capacities: not waited for yet
    assert_same(ta.export(), oracle.count(a).glob(), f"{slots} slots")
    assert_same(tb.export(), oracle.count(b).glob(), f"{slots} slots")
    assert_same(merged.export(), oracle.count(a + b" " + b).glob(), f"merged from {slots} slots")
    for t in (ta, tb, merged):
        t.free()


@pytest.mark.parametrize("ndocs", [400, 1100])
def test_documents_split_into_ranges(ctr, ndocs):
    docs = [text(5_200 + 7 * d % 500, d) for d in range(200)]
    docs = [docs[d % 200] for d in range(ndocs)]
    assert min(len(d) for d in docs) > 64 << 10
    data = np.frombuffer(b"\n".join(docs) + b"\n", np.uint8).copy()
    offs = np.cumsum([0] + [len(d) + 1 for d in docs]).astype(np.uint64)
    b, keep = run_batched(ctr, data, offs, checked=True)
    check_docs(b, oracle.count(data, offs), ndocs)
    b.free()
