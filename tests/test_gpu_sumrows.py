"""The sum-row tile (csrc/sumrows.h): packed copies of integer input on plans
where neighbouring trial DMs and channels share most of their shift
differences.  Bit-exact against the oracle at the edges of its tiles: one DM,
a block of 128 DMs and one more, outputs that end in either half of a 736-word
time tile, groups of odd size, bins, saturated input (every 16-bit lane gives
up its high bytes), channels out of frequency order, and a delay span of more
than one pass of the row builders."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from synth import channel_freqs, filterbank, filterbank4

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _input(dtype, n_chan, n_samp, seed, full=False):
    if dtype == "u4":
        data = filterbank4(n_chan, n_samp, seed, 8.0, 4.0, row_bytes=(n_samp + 31) // 32 * 16)
        if full:
            data[:] = 255
        return oracle.Packed4(data, n_samp), torch.from_numpy(data).cuda()
    npdt, mean, sd, top = {"u8": (np.uint8, 128, 60, 255),
                           "u16": (np.uint16, 40000, 12000, 65535)}[dtype]
    x = filterbank(npdt, n_chan, n_samp, seed, mean, sd)
    if full:
        x[:] = top
    stride = (n_samp + 15) // 16 * 16
    xd = torch.full((n_chan, stride), top, dtype=torch.int32, device="cuda")
    xd[:, :n_samp] = torch.from_numpy(x.astype(np.int32)).cuda()
    return x, xd.to(torch.uint8 if dtype == "u8" else torch.uint16)


# dtype, channels, DMs, step (delay per trial at the lowest channel, samples), extra outputs, bin, full
CASES = [
    ("u8", 600, 1, 0.5, 1, 1, False),
    ("u8", 600, 127, 0.1, 367, 1, False),
    ("u8", 601, 128, 0.1, 368, 1, False),
    ("u8", 601, 129, 0.1, 369, 1, False),
    ("u8", 777, 257, 0.2, 735, 1, False),
    ("u8", 777, 300, 0.3, 736, 1, True),
    ("u8", 1024, 256, 0.6, 1472, 1, True),
    ("u8", 2048, 256, 1.2, 2209, 1, False),
    ("u8", 4099, 128, 2.5, 1473, 1, False),   # rows of more than 640 words: two passes
    ("u8", 513, 200, 0.2, 1841, 2, True),
    ("u8", 513, 200, 0.2, 1105, 4, True),
    ("u8", 513, 200, 0.2, 1000, 8, True),
    ("u4", 700, 200, 0.2, 1500, 1, True),
    ("u4", 700, 200, 0.2, 1105, 1, False),
    ("u16", 600, 130, 0.1, 1, 1, False),
    ("u16", 600, 130, 0.1, 369, 1, True),
    ("u16", 1000, 256, 0.5, 1105, 1, False),
]


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,extra,bin_,full", CASES)
def test_sum_row_tile_matches_oracle(dtype, n_chan, n_dm, slope, extra, bin_, full):
    f_high, t_samp = 1500.0, 64e-6
    freqs = channel_freqs(f_high, 300.0, n_chan)
    step = slope * bin_ * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    ranges = [(0.0, n_dm * step, step, bin_)]
    s_max = oracle.extent(freqs, f_high, t_samp, ranges[0], 10 ** 9)[0]
    n_samp = (s_max + extra) * bin_ + (bin_ - 1)
    x, xd = _input(dtype, n_chan, n_samp, 7100 + n_chan + n_dm, full)
    ref = oracle.forward(x, freqs, f_high, t_samp, ranges)[0]
    plan = dd.Plan(freqs, f_high, t_samp, ranges, dtype)
    if not plan.info(n_samp)["packed_copy"][0]:
        plan.set_tile(0, "packed")
    for segments in (1, 3):
        got = plan.run(xd, n_samp=n_samp, segments=segments)[0].cpu().numpy()
        plan.device_status()
        np.testing.assert_array_equal(got, ref, err_msg=f"segments {segments}")


def test_sum_row_tile_with_channels_out_of_order():
    """Channel differences of either sign (neighbours swapped) and a DM range
    that does not start at zero."""
    rng = np.random.default_rng(7300)
    freqs = channel_freqs(1500.0, 300.0, 1200)
    order = np.arange(1200)
    for i in range(0, 1199, 2):
        if rng.random() < 0.5:
            order[[i, i + 1]] = order[[i + 1, i]]
    freqs = np.ascontiguousarray(freqs[order])
    step = 0.3 * 64e-6 / oracle.delay_coeff(freqs.min(), 1500.0)
    ranges = [(40 * step, 300 * step, step, 1)]
    n_samp = 4001
    x, xd = _input("u8", 1200, n_samp, 7301)
    ref = oracle.forward(x, freqs, 1500.0, 64e-6, ranges)[0]
    plan = dd.Plan(freqs, 1500.0, 64e-6, ranges, "u8")
    got = plan.run(xd, n_samp=n_samp, segments=1)[0].cpu().numpy()
    np.testing.assert_array_equal(got, ref)


def test_sum_row_tile_windows_and_withheld_group():
    """A window's compact rows; and a group whose copies never come: the waits
    run out, the status word says so, nothing hangs, and the next run is exact."""
    freqs = channel_freqs(1500.0, 300.0, 640)
    step = 0.2 * 64e-6 / oracle.delay_coeff(freqs[-1], 1500.0)
    ranges = [(0.0, 200 * step, step, 1)]
    n_samp = 6000
    x, xd = _input("u8", 640, n_samp, 7400)
    ref = oracle.forward(x, freqs, 1500.0, 64e-6, ranges)[0]
    plan = dd.Plan(freqs, 1500.0, 64e-6, ranges, "u8")
    plan.set_tile(0, "packed")
    for keep in (1, 368, 737, 1500):
        got = plan.run_window(xd, [keep], n_samp=n_samp)[0].cpu().numpy()
        np.testing.assert_array_equal(got, ref[:, :keep], err_msg=f"keep {keep}")
    for hold in (0, 1, 2, 5):
        plan.set_wait_limit(2000, hold)
        plan.run(xd, n_samp=n_samp, segments=1)
        torch.cuda.synchronize()
        with pytest.raises(dd.DDError):
            plan.device_status()
        plan.set_wait_limit(0, -1)
        got = plan.run(xd, n_samp=n_samp, segments=1)[0].cpu().numpy()
        plan.device_status()
        np.testing.assert_array_equal(got, ref, err_msg=f"after holding group {hold}")


# dtype, channels, DMs, slope, extra outputs, full
RAW_CASES = [
    ("u8", 600, 1, 0.5, 1, False), ("u8", 601, 129, 0.1, 736, True),
    ("u8", 777, 257, 0.2, 737, False), ("u8", 1024, 256, 0.6, 1473, True),
    ("u8", 2048, 256, 1.2, 2209, False), ("u8", 4099, 128, 2.5, 1473, False),
    ("u4", 700, 200, 0.2, 735, True), ("u4", 703, 129, 0.15, 1841, False),
    ("u4", 4099, 128, 2.5, 737, False),
    ("u16", 600, 130, 0.1, 368, False), ("u16", 1000, 256, 0.5, 1105, True),
    ("u16", 4099, 128, 2.5, 737, False),
]


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,extra,full", RAW_CASES)
def test_sum_row_tile_from_the_input(dtype, n_chan, n_dm, slope, extra, full):
    """Without scratch, alone and in a batch of two beams (the persistent
    kernel, several items per CTA slot), against the oracle."""
    from paper_2311_05341_gb300 import batch
    f_high, t_samp = 1500.0, 64e-6
    freqs = channel_freqs(f_high, 300.0, n_chan)
    step = slope * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    ranges = [(0.0, n_dm * step, step, 1)]
    s_max = oracle.extent(freqs, f_high, t_samp, ranges[0], 10 ** 9)[0]
    n_samp = s_max + extra
    x, xd = _input(dtype, n_chan, n_samp, 7500 + n_chan + n_dm, full)
    ref = oracle.forward(x, freqs, f_high, t_samp, ranges)[0]
    plan = dd.Plan(freqs, f_high, t_samp, ranges, dtype)
    got = plan.run(xd, n_samp=n_samp, segments=0)[0].cpu().numpy()
    plan.device_status()
    np.testing.assert_array_equal(got, ref)
    beams = [batch.BeamSpec(freqs, f_high, t_samp, ranges, dtype, n_samp)] * 2
    runner = batch.BatchRunner(beams, autotune=False, graph=False,
                               tiles=[[("pattern", -1)], [("packed", -1)]])
    for t in runner.inputs:
        t[:, :xd.shape[1]].copy_(xd[:, :t.shape[1]])
    for _ in range(2):
        runner.run()
        runner.status()
        for i in range(2):
            np.testing.assert_array_equal(runner.planes(i)[0].cpu().numpy(), ref)


@pytest.mark.parametrize("n_chan,n_dm,slope,extra,full", [
    (513, 200, 0.2, 1841, True), (1000, 129, 0.15, 735, False), (2047, 256, 0.9, 737, True),
    (600, 1, 0.5, 1, False)])
def test_sum_row_tile_decimates_the_input_by_two(n_chan, n_dm, slope, extra, full):
    """Bin 2 from the input: alone, as a window, through the segmented host
    pipeline (segments start at multiples of 736 outputs) and in a batch."""
    from paper_2311_05341_gb300 import batch
    f_high, t_samp = 1500.0, 64e-6
    freqs = channel_freqs(f_high, 300.0, n_chan)
    step = slope * 2 * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    ranges = [(0.0, n_dm * step, step, 2)]
    s_max = oracle.extent(freqs, f_high, t_samp, ranges[0], 10 ** 9)[0]
    n_samp = 2 * (s_max + extra) + 1
    x, xd = _input("u8", n_chan, n_samp, 7700 + n_chan, full)
    ref = oracle.forward(x, freqs, f_high, t_samp, ranges)[0]
    plan = dd.Plan(freqs, f_high, t_samp, ranges, "u8")
    got = plan.run(xd, n_samp=n_samp)[0].cpu().numpy()
    plan.device_status()
    np.testing.assert_array_equal(got, ref)
    keep = max(1, extra // 2)
    got = plan.run_window(xd, [keep], n_samp=n_samp)[0].cpu().numpy()
    np.testing.assert_array_equal(got, ref[:, :keep])
    h_in, d_out = xd.cpu().pin_memory(), plan.empty_output(n_samp)
    h_out = torch.full(d_out.shape, -1, dtype=d_out.dtype).pin_memory()
    plan.run_host(h_in, h_out, torch.zeros_like(xd), d_out, n_samp=n_samp)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(plan.split(h_out, n_samp)[0].numpy(), ref)
    runner = batch.BatchRunner([batch.BeamSpec(freqs, f_high, t_samp, ranges, "u8", n_samp)],
                               autotune=False, graph=False)
    runner.inputs[0][:, :xd.shape[1]].copy_(xd[:, :runner.inputs[0].shape[1]])
    runner.run()
    runner.status()
    np.testing.assert_array_equal(runner.planes(0)[0].cpu().numpy(), ref)
