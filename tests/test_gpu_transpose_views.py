"""transpose of a column block of a wider time-major array, up to the array's
last byte: no piece beyond the block's channels is read."""
import numpy as np
import pytest

import paper_2311_05341_gb300 as dd

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("blocks,first,n_chan", [(15, 8, 112), (15, 14, 5), (9, 0, 129), (20, 3, 130)])
def test_column_block(dtype, blocks, first, n_chan):
    per = 16 // np.dtype(dtype).itemsize
    width, c0 = blocks * per, first * per
    n_chan = min(n_chan, width - c0)
    x = np.random.default_rng(blocks).integers(1, 250, (301, width)).astype(dtype)
    view = torch.from_numpy(x).cuda()[:, c0:]
    got = dd.transpose(view, n_chan=n_chan).cpu().numpy()
    np.testing.assert_array_equal(got[:, :301], x[:, c0:c0 + n_chan].T)
    assert not got[:, 301:].any()
