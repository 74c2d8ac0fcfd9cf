"""Merging top-k tables whose source holds as many words of 17+ letters as they
keep rows: the merge is sized by the rows themselves.  Against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,kept_long", [(3000, 0), (3000, 40), (5, 0)])
def test_merge_of_topk_tables(k, kept_long):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    tops, want = [], {}
    for seed in (1, 2):
        rng = np.random.default_rng(seed)

        def words(n, lo, hi):
            out = set()
            while len(out) < n:
                out.add(bytes(rng.integers(97, 123, int(rng.integers(lo, hi + 1))).astype(np.uint8)))
            return sorted(out)
        short, long_ = words(k - kept_long, 5, 14), words(k, 17, 30)
        kept = short + long_[:kept_long]  # twice each, the other long words once
        text = b" ".join(kept * 2 + long_[kept_long:])
        table = ctr.count_checked(to_dev(text))
        top = ctr.topk(table, k)
        rows = top.as_list()  # waits: the merge knows its sizes
        assert sorted(rows) == sorted((w, 2) for w in kept)
        for w, c in rows:
            want[w] = want.get(w, 0) + c
        tops.append(top)
    merged = ctr.merge(tops)
    want = sorted(want.items(), key=lambda x: (-x[1], x[0]))
    assert_same(merged.export(), oracle.Table.from_list(want), "merged")
    again = ctr.merge([merged, tops[0]])
    assert len(again.as_list()) == len(want)
    ctr.close()
