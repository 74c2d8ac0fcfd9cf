"""wc_row_sums at every alignment of a row's first word and at the edges of its
16-byte groups and of a warp's round of loads (1,024 words): whole numbers,
equal to the host's sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 2, 3, 4, 5, 7, 9, 127, 128, 131, 1023, 1024, 1027, 2050, 4099])
@pytest.mark.parametrize("skip", [0, 1, 2, 3])
def test_row_sums_alignments(cols, skip):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_05269_gb300 import wc
    rows = 37
    rng = np.random.default_rng(cols * 4 + skip)
    m = rng.integers(0, 1 << 32, size=(rows, cols), dtype=np.uint64).astype(np.uint32)
    buf = torch.full((skip + rows * cols + 8,), -1, dtype=torch.int32, device="cuda:0")  # all ones around the matrix
    buf[skip:skip + rows * cols] = torch.from_numpy(m.reshape(-1).view(np.int32)).to("cuda:0")
    out = torch.full((rows,), -1, dtype=torch.int64, device="cuda:0")
    wc.wc_row_sums(buf.data_ptr() + 4 * skip, rows, cols, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), m.astype(np.uint64).sum(axis=1))
