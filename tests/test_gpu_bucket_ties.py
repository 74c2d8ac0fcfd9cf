"""The bucket sort where a word of 16 letters and a longer one that begins with
it are counted equally often and are both sampled: each is told apart from the
other, wherever the longer one sits in its hash table (its first slot among
them: 60 long words in 64 slots).  Few entries in many slots, so that every one
is sampled; a varying number of words before them puts either of a pair where a
splitter is taken.  Against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("before", range(6))
def test_words_behind_their_prefix(before):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    for seed in range(4):
        rng = np.random.default_rng(10 * before + seed)
        prefix = [bytes(rng.integers(97, 123, 16).astype(np.uint8)) for _ in range(60)]
        words = prefix + [p + bytes(rng.integers(97, 123, 1 + i % 20).astype(np.uint8)) for i, p in enumerate(prefix)]
        words += [b"%c" % (97 + i) for i in range(before)] * 2
        rng.shuffle(words)
        text = b" ".join(words)
        got = ctr.count(to_dev(text), opts=(1 << 15, 64, 1 << 16))
        assert_same(got.export(), oracle.count(text).glob(), f"{before} before, {seed}")
        got.free()
    ctr.close()
