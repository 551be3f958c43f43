"""The sum-row kernels' waits that run out: a channel group whose copies never
come, in every window format and in the persistent batch kernel.  Adding and
building warps of a CTA give up at different points of their pipeline; the
status word says so, every warp leaves, the copies in flight land, and the next
run is exact."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import _lib
from paper_2311_05341_gb300 import batch as ddb
from synth import channel_freqs, filterbank, filterbank4

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

POLLS = 2000
F_HIGH, T_SAMP = 1500.0, 64e-6


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _input(dtype, n_chan, n_samp, seed):
    if dtype == "u4":
        data = filterbank4(n_chan, n_samp, seed, 8.0, 4.0, row_bytes=(n_samp + 31) // 32 * 16)
        return oracle.Packed4(data, n_samp), torch.from_numpy(data).cuda()
    npdt, mean, sd = {"u8": (np.uint8, 128, 60), "u16": (np.uint16, 40000, 9000)}[dtype]
    x = filterbank(npdt, n_chan, n_samp, seed, mean, sd)
    xd = torch.zeros((n_chan, (n_samp + 15) // 16 * 16), dtype=getattr(torch, str(x.dtype)),
                     device="cuda")
    xd[:, :n_samp].copy_(torch.from_numpy(x).cuda())
    return x, xd


def _ranges(n_chan, n_dm, slope, bin_=1):
    freqs = channel_freqs(F_HIGH, 300.0, n_chan)
    step = slope * bin_ * T_SAMP / oracle.delay_coeff(freqs[-1], F_HIGH)
    return freqs, [(0.0, n_dm * step, step, bin_)]


# dtype, channels, DMs, samples, bin, segments of Plan.run (0: from the input)
FORMS = [("u8", 640, 200, 6000, 1, 0), ("u8", 640, 200, 6000, 1, 3), ("u4", 700, 200, 6000, 1, 0),
         ("u16", 600, 200, 6000, 1, 0), ("u8", 500, 1024, 2 * 13000, 2, 0)]


@pytest.mark.parametrize("dtype,n_chan,n_dm,n_samp,bin_,segments", FORMS)
def test_withheld_group_in_every_form(dtype, n_chan, n_dm, n_samp, bin_, segments):
    freqs, ranges = _ranges(n_chan, n_dm, 0.2, bin_)
    x, xd = _input(dtype, n_chan, n_samp, 9100 + n_chan)
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, dtype)
    ref = oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0]
    for hold in (0, 1, 3, 8):
        plan.set_wait_limit(POLLS, hold)
        plan.run(xd, n_samp=n_samp, segments=segments)
        torch.cuda.synchronize()  # the kernels returned
        with pytest.raises(dd.DDError) as ei:
            plan.device_status()
        assert ei.value.status == _lib.DD_ERR_TIMEOUT
        plan.set_wait_limit(0, -1)
        got = plan.run(xd, n_samp=n_samp, segments=segments)[0].cpu().numpy()
        plan.device_status()
        np.testing.assert_array_equal(got, ref, err_msg=f"after holding group {hold}")


@pytest.mark.parametrize("dtype,tile", [("u8", "pattern"), ("u8", "packed"), ("u4", "pattern"),
                                        ("u16", "pattern")])
def test_withheld_group_in_a_batch(dtype, tile):
    freqs, ranges = _ranges(640, 200, 0.2)
    beams = [ddb.BeamSpec(freqs, F_HIGH, T_SAMP, ranges, dtype, n) for n in (9000, 7000)]
    runner = ddb.BatchRunner(beams, autotune=False, graph=False, tiles=[[(tile, -1)], [(tile, -1)]])
    refs = []
    for i, (b, t) in enumerate(zip(beams, runner.inputs)):
        x, xd = _input(dtype, 640, b.n_samp, 9200 + i)
        w = min(t.shape[1], xd.shape[1])
        t[:, :w].copy_(xd[:, :w])
        refs.append(oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0])
    for hold in (0, 2, 7):
        runner.plans[1].set_wait_limit(POLLS, hold)
        runner.bind()
        runner.run()
        torch.cuda.synchronize()
        with pytest.raises(dd.DDError) as ei:
            runner.status()
        assert ei.value.status == _lib.DD_ERR_TIMEOUT
        runner.plans[1].set_wait_limit(0, -1)
        runner.bind()
        runner.run()
        runner.status()
        for i in range(2):
            np.testing.assert_array_equal(runner.planes(i)[0].cpu().numpy(), refs[i])


@pytest.mark.parametrize("tile", ["pattern", "packed"])
def test_short_wait_limit_leaves_a_healthy_run_alone(tile):
    """64 polls of a copy's barrier suspend for longer than any copy takes, and
    the limit counts no other wait: an ordinary run keeps within it."""
    freqs, ranges = _ranges(640, 200, 0.2)
    x, xd = _input("u8", 640, 30000, 9300)
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, "u8")
    plan.set_tile(0, tile)
    plan.set_wait_limit(64, -1)
    got = plan.run(xd, n_samp=30000, segments=0)[0].cpu().numpy()
    plan.device_status()
    np.testing.assert_array_equal(got, oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0])
