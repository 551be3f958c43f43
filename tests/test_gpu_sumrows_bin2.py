"""uint8 at bin 2 from the input on the sum-row tile's one-unit kernel: launches
long enough that it is the one taken (asserted), whole, as a window and as the
segments of the host pipeline, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from synth import channel_freqs, filterbank

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

F_HIGH, T_SAMP = 1500.0, 64e-6


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _case(n_chan, n_dm, slope, n_out, seed, full):
    freqs = channel_freqs(F_HIGH, 300.0, n_chan)
    step = slope * 2 * T_SAMP / oracle.delay_coeff(freqs[-1], F_HIGH)
    ranges = [(0.0, n_dm * step, step, 2)]
    s_max = oracle.extent(freqs, F_HIGH, T_SAMP, ranges[0], 10 ** 9)[0]
    n_samp = 2 * (s_max + n_out) + 1
    x = filterbank(np.uint8, n_chan, n_samp, seed, 128, 60)
    if full:
        x[:] = 255
    xd = torch.full((n_chan, (n_samp + 15) // 16 * 16), 255, dtype=torch.uint8, device="cuda")
    xd[:, :n_samp].copy_(torch.from_numpy(x))
    return (dd.Plan(freqs, F_HIGH, T_SAMP, ranges, "u8"), n_samp, xd,
            oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0])


# Outputs at the edges of the 736-output units; every 16-bit lane gives up its
# high bytes where the input is saturated (513 channels of 510).
@pytest.mark.parametrize("n_chan,n_dm,slope,n_out,full", [
    (200, 1024, 0.1, 736 * 18, False), (513, 1023, 0.2, 736 * 20 + 1, True),
    (301, 1150, 0.15, 736 * 17 - 1, False)])
def test_whole_and_window(n_chan, n_dm, slope, n_out, full):
    plan, n_samp, xd, ref = _case(n_chan, n_dm, slope, n_out, 9500 + n_chan, full)
    for keep in (ref.shape[1], 736 * 15 + 5):
        assert plan.run_kernel(0, keep) == ("sum-rows", False)
        got = plan.run_window(xd, [keep], n_samp=n_samp)[0].cpu().numpy()
        plan.device_status()
        np.testing.assert_array_equal(got, ref[:, :keep], err_msg=f"keep {keep}")


def test_segments_of_the_host_pipeline():
    """Segments start at multiples of 736 outputs past 0; the last one, short,
    may take either kernel."""
    plan, n_samp, xd, ref = _case(200, 1024, 0.1, 200001, 9600, False)
    seg = (n_samp + 15) // 16 // 2 // 736 * 736 - 736
    assert plan.run_kernel(0, seg) == ("sum-rows", False)
    h_in, d_out = xd.cpu().pin_memory(), plan.empty_output(n_samp)
    h_out = torch.full(d_out.shape, -1, dtype=d_out.dtype).pin_memory()
    plan.run_host(h_in, h_out, torch.zeros_like(xd), d_out, n_samp=n_samp)
    torch.cuda.synchronize()
    plan.device_status()
    np.testing.assert_array_equal(plan.split(h_out, n_samp)[0].numpy(), ref)
