"""Calls inside a stream capture, after calls outside it whose freed memory the
context still watches: the capture stays valid, the graph replays, and the
bytes come off the charge."""
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_series_sum_captured_after_a_warm_up(mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    out = torch.zeros(2, dtype=torch.float64, device="cuda:0")
    side = torch.cuda.Stream()

    def both(n, stream):
        for k, series in enumerate((wc.WC_SERIES_SQRT, wc.WC_SERIES_ALT_HARMONIC)):
            wc.wc_series_sum(ctr.ctx, series, n, out.data_ptr() + 8 * k, stream.cuda_stream)

    with torch.cuda.stream(side):
        both(1000, side)  # leaves freed memory to be seen done
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode=mode):
        both(300_007, side)
        used, _ = wc.wc_mem_usage(ctr.ctx)  # (reads no stream)
    assert used == 0
    out.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    want = [oracle.series_sum(s, 300_007) for s in (wc.WC_SERIES_SQRT, wc.WC_SERIES_ALT_HARMONIC)]
    # the oracle's compensated sums are within 2.2e-16 of the sum, the kernel's within 1.1e-16
    assert out.cpu().tolist() == pytest.approx(want, rel=1e-15, abs=0)
    assert wc.wc_mem_usage(ctr.ctx)[0] == 0
    del graph
    ctr.close()
