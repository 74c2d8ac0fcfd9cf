"""Batches so large that documents of a little over 64 KB are counted whole by
one block, where these documents hold more distinct words (11,600) or more
distinct words of 17+ letters (95) than a block's tables take: all their words
go to the (document, word) tables, which must have room for them, in a plan as
in a single call.  Against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_batched import check_docs

pytestmark = pytest.mark.gpu

SIZE, FILLER = 70_000, 64_000  # bytes; the filler documents hold one word


def rich(seed: int) -> bytes:
    """Distinct words of five letters."""
    n = np.random.default_rng(seed).choice(26 ** 5, SIZE // 6, replace=False)
    w = np.full((n.size, 6), ord(" "), np.uint8)
    for j in range(5):
        w[:, j] = 97 + n // 26 ** j % 26
    return w.tobytes()


def many_long(seed: int) -> bytes:
    rng = np.random.default_rng(seed)
    w = [bytes(rng.integers(97, 123, 17 + i % 4).astype(np.uint8)) for i in range(95)]
    return b" ".join([x + b" a b a c" * 20 for x in w])


def test_whole_documents_past_the_blocks_tables():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    docs = [rich(d) for d in range(110)] + [(many_long(d) * 5)[:SIZE - 1] + b" " for d in range(180)]
    # a document is kept whole up to a sixteenth of an even share of the batch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    fill = 16 * sms * (SIZE + 2_000) // FILLER
    sizes = [len(d) for d in docs] + [FILLER] * fill
    offs = np.cumsum([0] + sizes).astype(np.uint64)
    text = np.concatenate([np.frombuffer(b"".join(docs), np.uint8), np.tile(np.frombuffer(b"z ", np.uint8), FILLER // 2 * fill)])
    assert text.size == int(offs[-1])
    dev = torch.device("cuda:0")
    t, o = torch.from_numpy(text).to(dev), torch.from_numpy(offs.view(np.int64)).to(dev)
    r = oracle.count(text[:int(offs[len(docs)])], offs[:len(docs) + 1])
    ctr = wc.Counter(0, count_bits=32)
    plan = ctr.plan(offs, 0)
    single = ctr.count_batched(t, o, offs)
    for b in (single, plan.run(t, o)):
        check_docs(b, r, len(docs))
        ds, dn, w, wo, c = b.export()
        assert (dn[len(docs):] == 1).all() and (c[ds[len(docs):]] == FILLER // 2).all()
    plan.free()
    single.free()
    ctr.close()
