"""GPU parity of long texts (1 KB strips; from 80 MB on with a sampled head)
against the oracle: words of every length at every place of a strip, dense and
empty stretches, runs longer than a strip, unaligned bases and ends, both sides
of the sizes where the strips and the head change."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu

WIDE, HEAD = 16 << 20, 80 << 20


@pytest.fixture(scope="module")
def ctr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    c = wc.Counter(0)
    yield c
    c.close()


def block() -> np.ndarray:
    """About 1 MB whose length shares no factor with a strip, so that its
    repetitions meet the strips at ever other places."""
    rng = np.random.default_rng(5)
    vocab = [bytes(rng.integers(97, 123, n).astype(np.uint8)) for n in list(range(1, 41)) * 40]
    out, seps = [], [b" ", b". ", b"\n", b" 17 ", b"-", b"\xc3\xa9"]
    for i in (rng.zipf(1.2, 110_000) * 7) % len(vocab):
        w = vocab[i]
        out.append(w.upper() if i % 5 == 0 else w)
        out.append(seps[int(rng.integers(0, len(seps)))])
    text = b"".join(out)[:900_000]
    text += b"a b " * 1500 + b"\x00" * 3000 + b" " + b"q" * 3001 + b" " + rng.integers(0, 256, 20_000).astype(np.uint8).tobytes()
    text += b" " * (1_000_003 - len(text)) if len(text) < 1_000_003 else b""
    return np.frombuffer(text[:1_000_003], dtype=np.uint8)


@pytest.mark.parametrize("n,offset", [(WIDE - 1, 0), (WIDE, 3), (WIDE + 1023, 16), (WIDE + 5_000_017, 9), (HEAD - 1, 1),
                                      (HEAD, 0), (HEAD + 3_333_333, 13)])
def test_long_text(ctr, n, offset):
    b = block()
    text = np.tile(b, n // b.size + 1)[:n]
    want = oracle.count(text).glob()
    assert_same(ctr.count_checked(to_dev(text.tobytes(), offset)).export(), want, f"{n} at {offset}")
