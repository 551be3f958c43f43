"""The time-major transpose at the edges of its 128-byte x 256-byte tiles:
windows that start off the 16-byte grid (written word by word), one sample
more and less than a tile, and an output made by the call, whose row padding
is zero."""
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
@pytest.mark.parametrize("n_samp,n_chan,t_begin,t_end", [
    (255, 127, 0, None), (256, 128, 0, None), (257, 129, 0, None), (513, 33, 4, 513),
    (700, 300, 4, 261), (700, 300, 260, 700), (64, 31, 8, 8), (65, 65, 0, 64)])
def test_transpose_edges(dtype, n_samp, n_chan, t_begin, t_end):
    per = 16 // np.dtype(dtype).itemsize
    rng = np.random.default_rng(n_samp + n_chan)
    x = rng.integers(1, 250, (n_samp, (n_chan + per - 1) // per * per)).astype(dtype)
    got = dd.transpose(torch.from_numpy(x).cuda(), n_chan=n_chan, t_begin=t_begin, t_end=t_end)
    ref = np.zeros((n_chan, (n_samp + per - 1) // per * per), dtype)
    te = n_samp if t_end is None else t_end
    ref[:, t_begin:te] = x[t_begin:te, :n_chan].T
    np.testing.assert_array_equal(got.cpu().numpy(), ref)
