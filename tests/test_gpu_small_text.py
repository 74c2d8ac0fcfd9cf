"""GPU parity of short texts (one block counts, sorts and writes the table)
against the oracle and against the general path (reached by passing capacities),
around the sizes where the block's pieces, slots and its limit change."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu

LIMIT = 16384  # longest text counted by one block


@pytest.fixture(scope="module")
def ctr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    c = wc.Counter(0)
    yield c
    c.close()


def text(kind: str, n: int) -> bytes:
    rng = np.random.default_rng(n + len(kind))
    if kind == "one":  # one word, as long as the text
        return b"q" * n
    if kind == "letters":  # as many words as fit
        return (b"a " * (n // 2 + 1))[:n]
    if kind == "distinct":  # as many distinct words as fit
        al = [bytes([c]) for c in range(97, 123)]
        ws = al + [a + b for a in al for b in al] + [a + b + c for a in al for b in al for c in al]
        return b" ".join(ws[:n // 2 + 1])[:n]
    if kind == "ties":  # equal counts, long words that share 16 letters and more
        ws = [b"z" * k + bytes(rng.integers(97, 100, int(rng.integers(0, 40))).astype(np.uint8))
              for k in (15, 16, 17, 31, 32, 33, 48) for _ in range(60)]
        return b"-".join(ws * 2)[:n]
    if kind == "bytes":  # any byte value
        return rng.integers(0, 256, n).astype(np.uint8).tobytes()
    w = rng.zipf(1.3, n) % 3000  # "zipf": ordinary words, both cases, varying separators
    ws = [b"w" + bytes((97 + int(x) // 26 ** k % 26) ^ (32 * int(x & 1)) for k in range(1 + int(x) % 9)) for x in w]
    return (b". ".join(ws) + b" ")[:n]


@pytest.mark.parametrize("kind", ["one", "letters", "distinct", "ties", "bytes", "zipf"])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 2047, 2049, 4097, LIMIT - 17, LIMIT - 1, LIMIT, LIMIT + 1])
def test_short_text(ctr, kind, n):
    data = text(kind, n)
    want = oracle.count(data).glob()
    for off in (0, 1, 15):
        t = ctr.count_checked(to_dev(data, off))
        g = ctr.count(to_dev(data, off), opts=(65536, 65536, 1 << 18))
        got = t.export()
        assert_same(got, want, f"{kind} {n} at {off}")
        assert_same(g.export(), want, f"{kind} {n} at {off}, general path")
        assert int(got[2].sum()) == int(want.counts.sum())
        both = ctr.merge([t, g])
        assert_same(both.export(), oracle.Table.from_list([(w, 2 * c) for w, c in want.as_list()]), "merged")
