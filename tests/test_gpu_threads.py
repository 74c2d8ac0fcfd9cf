"""Memory and tables of one context given back by other threads than the one that
counts with it (a garbage collector frees where it happens to run): the charge
comes back to zero and the counts stay right."""
import threading

import pytest

import oracle
from gpu_util import assert_same, to_dev

pytestmark = pytest.mark.gpu


def test_frees_from_other_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    failed = []

    def churn(stream):
        try:
            for i in range(1500):
                p = wc.wc_buffer_alloc(ctr.ctx, 4096 + i, stream.cuda_stream)
                wc.wc_buffer_free(ctr.ctx, p, 4096 + i, stream.cuda_stream)
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=churn, args=(torch.cuda.Stream(),)) for _ in range(4)]
    for t in threads:
        t.start()
    text = b"one two two three three three " * 2000
    want = oracle.count(text).glob()
    dev = to_dev(text)
    while any(t.is_alive() for t in threads):
        table = ctr.count_checked(dev)
        assert_same(table.export(), want, "beside other threads' frees")
        other = threading.Thread(target=table.free)
        other.start()
        other.join()
    for t in threads:
        t.join()
    assert not failed
    torch.cuda.synchronize()
    assert ctr.mem_usage()[0] == 0
    ctr.close()
