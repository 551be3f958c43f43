"""The output that transpose makes itself: small and large (zeroed whole, or the
rows' padding alone), on the current and on another stream."""
import numpy as np
import pytest

import paper_2311_05341_gb300 as dd

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n_chan,n_samp", [(65, 1001), (1024, 60001), (1024, 60000), (1030, 60015)])
@pytest.mark.parametrize("side", [False, True])
def test_made_output_is_padded_with_zeros(n_chan, n_samp, side):
    g = torch.Generator(device="cuda").manual_seed(n_samp)
    x = torch.randint(1, 256, (n_samp, (n_chan + 15) // 16 * 16), generator=g, device="cuda",
                      dtype=torch.int32).to(torch.uint8)
    width = (n_samp + 15) // 16 * 16
    want = torch.zeros((n_chan, width), dtype=torch.uint8, device="cuda")
    want[:, :n_samp] = x[:, :n_chan].t()
    # Freed memory of the same size holds other bytes.
    torch.full((n_chan, width), 170, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side else None
    got = dd.transpose(x, n_chan=n_chan, stream=stream)
    torch.cuda.synchronize()
    assert got.shape == (n_chan, width) and torch.equal(got, want)


@pytest.mark.parametrize("n_chan,n_samp,zeroed", [
    (64, 1001, True), (64, 1008, False), (1024, 32001, True), (1024, 65537, False)])
def test_small_outputs_are_zeroed_whole(monkeypatch, n_chan, n_samp, zeroed):
    """Zeroing the padding of a small output alone costs more than it saves."""
    x = torch.zeros((n_samp, n_chan), dtype=torch.uint8, device="cuda")
    calls, zeros = [], torch.zeros
    monkeypatch.setattr(torch, "zeros", lambda *a, **k: calls.append(a) or zeros(*a, **k))
    dd.transpose(x)
    assert len(calls) == zeroed
