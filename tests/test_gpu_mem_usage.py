"""The peak of wc_mem_usage leaves out memory whose free its stream has passed,
also while another stream's older free waits; thousands of waiting frees do not
hold up the host."""
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


def test_peak_beside_a_waiting_stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    slow, quick = torch.cuda.Stream(), torch.cuda.Stream()
    held = wc.wc_buffer_alloc(ctr.ctx, MB, slow.cuda_stream)
    torch.cuda.synchronize()
    ctr.mem_usage(reset=True)
    with torch.cuda.stream(slow):
        torch.cuda._sleep(1_000_000_000)  # about half a second
    wc.wc_buffer_free(ctr.ctx, held, MB, slow.cuda_stream)
    for _ in range(10):
        p = wc.wc_buffer_alloc(ctr.ctx, MB, quick.cuda_stream)
        wc.wc_buffer_free(ctr.ctx, p, MB, quick.cuda_stream)
        quick.synchronize()
    waiting = not slow.query()
    used, peak = ctr.mem_usage()
    assert waiting and used == MB, "the slow stream's work ended before the check"
    assert peak == 2 * MB
    torch.cuda.synchronize()
    assert ctr.mem_usage()[0] == 0
    ctr.close()


def test_thousands_of_waiting_frees():
    """Giving memory back takes microseconds; looking at every waiting free on
    every release took tenths of a millisecond."""
    import time

    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    ctr = wc.Counter(0)
    streams = [torch.cuda.Stream() for _ in range(8)]

    def host_seconds(n):
        t0 = time.perf_counter()
        for _ in range(n):
            for s in streams:
                p = wc.wc_buffer_alloc(ctr.ctx, 4096, s.cuda_stream)
                wc.wc_buffer_free(ctr.ctx, p, 4096, s.cuda_stream)
        return time.perf_counter() - t0

    host_seconds(350)  # pools and events made
    torch.cuda.synchronize()
    idle = host_seconds(350)
    torch.cuda.synchronize()
    for s in streams:
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000_000)  # about a second
    waiting = host_seconds(350)  # 2,800 frees
    assert not streams[0].query(), f"the streams' work ended before the host's ({waiting:.3f} s)"
    torch.cuda.synchronize()
    assert ctr.mem_usage()[0] == 0
    ctr.close()
    assert waiting < 4 * idle + 0.02, (waiting, idle)
