"""Steep plans on either side of the direct tile's rule, with a partial block of
DMs: the kernel the rule names, and the oracle's outputs."""
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


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,n_out,kernel", [
    ("f32", 33, 356, 8.0, 30001, "direct"), ("f32", 33, 400, 8.0, 16384, "offset"),
    ("u8", 40, 356, 7.0, 60002, "direct"), ("u8", 40, 400, 7.0, 32768, "offset"),
    ("u16", 21, 356, 6.0, 30003, "direct")])
def test_either_side_of_the_rule(dtype, n_chan, n_dm, slope, n_out, kernel):
    f_high, t_samp = 400.0, 327.68e-6
    freqs = channel_freqs(f_high, 100.0, n_chan)
    step = slope * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    ranges = [(0.0, n_dm * step, step, 1)]
    n_samp = oracle.extent(freqs, f_high, t_samp, ranges[0], 10 ** 9)[0] + n_out
    npdt, mean, sd = {"u8": (np.uint8, 128, 60), "u16": (np.uint16, 40000, 9000),
                      "f32": (np.float32, 0.0, 1.0)}[dtype]
    x = filterbank(npdt, n_chan, n_samp, 9700 + n_dm, mean, sd)
    per = 16 // x.itemsize
    xd = torch.zeros((n_chan, (n_samp + per - 1) // per * per), dtype=getattr(torch, str(x.dtype)),
                     device="cuda")
    xd[:, :n_samp].copy_(torch.from_numpy(x))
    plan = dd.Plan(freqs, f_high, t_samp, ranges, dtype)
    assert plan.run_kernel(0, n_out) == (kernel, False)
    got = plan.run(xd, n_samp=n_samp)[0].cpu().numpy()
    plan.device_status()
    ref = oracle.forward(x, freqs, f_high, t_samp, ranges)[0]
    if dtype == "f32":
        assert_float_parity(got, ref, oracle.forward(x, freqs, f_high, t_samp, ranges,
                                                     take_abs=True)[0])
    else:
        np.testing.assert_array_equal(got, ref)
