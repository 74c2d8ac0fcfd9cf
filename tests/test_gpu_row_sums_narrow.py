"""wc_row_sums on both sides of the width up to which rows are read word by word
(512), with fewer and more rows than resident warps: whole numbers, equal to the
host's sums.  Narrow rows take no longer than wide ones of the same bytes would
allow: a row of 31 words costs a few loads, not the 16-byte ones of a wide row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def device_matrix(rows, cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m = np.random.default_rng(rows + cols).integers(0, 1 << 32, size=(rows, cols), dtype=np.uint64).astype(np.uint32)
    return torch, m, torch.from_numpy(m.view(np.int32).reshape(-1)).to("cuda:0")


@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 96), (7, 97), (20_000, 1), (50_001, 33), (30_000, 129), (20_001, 511),
                                       (20_001, 512), (20_001, 513)])
def test_sums(rows, cols):
    from paper_2206_05269_gb300 import wc
    torch, m, d = device_matrix(rows, cols)
    out = torch.full((rows,), -1, dtype=torch.int64, device="cuda:0")
    wc.wc_row_sums(d.data_ptr(), rows, cols, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), m.astype(np.uint64).sum(axis=1))


def test_narrow_rows_are_not_slow():
    from paper_2206_05269_gb300 import wc
    torch, m, d = device_matrix(400_000, 31)
    out = torch.empty(400_000, dtype=torch.int64, device="cuda:0")
    best = 1e9
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        wc.wc_row_sums(d.data_ptr(), 400_000, 31, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    assert best < 0.09, best  # measured: 0.055 ms word by word, 0.127 by eight 16-byte loads a lane
