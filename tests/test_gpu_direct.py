"""The direct tile (csrc/direct.h): steep plans, more than 5 samples of delay
between consecutive trials, uint8 (bins 1, 2, 4), uint16 (1, 2) and float32, against the oracle; at
the edges of its blocks of 128 DMs and tiles of 368 words, with enough
channels for the 16-bit lanes to give up their high bytes."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from synth import channel_freqs, filterbank

from gpu_util import assert_float_parity

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# dtype, channels, DMs, samples of delay per trial, outputs, bin, saturated
# (enough outputs that the launch rule takes the direct tile)
CASES = [
    ("u8", 300, 128, 12.0, 150001, 1, False), ("u8", 520, 255, 6.0, 109665, 1, True),
    ("u8", 37, 300, 7.3, 36801, 2, True), ("u8", 100, 256, 11.0, 44161, 4, False),
    ("u16", 64, 200, 9.0, 44159, 1, True), ("u16", 21, 128, 6.1, 88321, 2, False),
    ("f32", 64, 128, 12.0, 88320, 1, False), ("f32", 5, 500, 20.0, 22081, 1, False),
    ("f32", 33, 257, 8.0, 30001, 1, False),
]


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,n_out,bin_,full", CASES)
def test_direct_tile_matches_oracle(dtype, n_chan, n_dm, slope, n_out, bin_, full):
    f_high, t_samp = 400.0, 327.68e-6
    freqs = channel_freqs(f_high, 100.0, n_chan)
    step = slope * bin_ * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    ranges = [(0.0, n_dm * step, step, bin_)]
    s_max = oracle.extent(freqs, f_high, t_samp, ranges[0], 10 ** 9)[0]
    n_samp = (s_max + n_out) * bin_ + bin_ - 1
    npdt, mean, sd, top = {"u8": (np.uint8, 128, 60, 255), "u16": (np.uint16, 40000, 9000, 65535),
                           "f32": (np.float32, 0.0, 1.0, 0)}[dtype]
    x = filterbank(npdt, n_chan, n_samp, 8100 + n_chan + n_dm, mean, sd)
    if full:
        x[:] = top
    per = 16 // x.itemsize
    xd = torch.zeros((n_chan, (n_samp + per - 1) // per * per), dtype=getattr(torch, str(x.dtype)),
                     device="cuda")
    xd[:, :n_samp].copy_(torch.from_numpy(x))
    ref = oracle.forward(x, freqs, f_high, t_samp, ranges)[0]
    plan = dd.Plan(freqs, f_high, t_samp, ranges, dtype)
    assert plan.info(n_samp)["tile_dms"][0] in (1, 2)
    got = plan.run(xd, n_samp=n_samp)[0].cpu().numpy()
    plan.device_status()
    if dtype == "f32":
        ab = oracle.forward(x, freqs, f_high, t_samp, ranges, take_abs=True)[0]
        assert_float_parity(got, ref, ab)
    else:
        np.testing.assert_array_equal(got, ref)


def test_direct_tile_withheld_stage():
    """A stage whose copies never come ends in the status word; then exact."""
    freqs = channel_freqs(400.0, 100.0, 100)
    step = 9.0 * 327.68e-6 / oracle.delay_coeff(freqs[-1], 400.0)
    n_samp = 90000
    for dtype, npdt in (("u8", np.uint8), ("f32", np.float32)):
        x = filterbank(npdt, 100, n_samp, 8200, 100.0, 20.0)
        xd = torch.from_numpy(x).cuda()
        plan = dd.Plan(freqs, 400.0, 327.68e-6, [(0.0, 256 * step, step, 1)], dtype)
        first = plan.run(xd)[0].clone()
        for hold in (0, 1, 3):
            plan.set_wait_limit(2000, hold)
            plan.run(xd)
            torch.cuda.synchronize()
            with pytest.raises(dd.DDError):
                plan.device_status()
            plan.set_wait_limit(0, -1)
            assert torch.equal(plan.run(xd)[0], first)
            plan.device_status()
