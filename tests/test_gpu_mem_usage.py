"""The peak of wc_mem_usage leaves out memory whose free its stream has passed,
also while another stream's older free waits."""
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
