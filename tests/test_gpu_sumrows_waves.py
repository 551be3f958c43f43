"""Launches of few waves, where the pattern tile takes over from the sum-row
tile: the oracle's outputs either way, alone, in the ring, in the host pipeline
and in batches, whose units tell which tile they run."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import batch as ddb
from synth import channel_freqs, filterbank, filterbank4

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

F_HIGH, T_SAMP = 1500.0, 64e-6


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _beam(dtype, n_chan, n_dm, slope, n_out, bin_=1):
    freqs = channel_freqs(F_HIGH, 300.0, n_chan)
    step = slope * bin_ * T_SAMP / oracle.delay_coeff(freqs[-1], F_HIGH)
    ranges = [(0.0, n_dm * step, step, bin_)]
    n_samp = (oracle.extent(freqs, F_HIGH, T_SAMP, ranges[0], 10 ** 9)[0] + n_out) * bin_
    if dtype == "u4":
        data = filterbank4(n_chan, n_samp, 9800, 8.0, 4.0, row_bytes=(n_samp + 31) // 32 * 16)
        x, xd = oracle.Packed4(data, n_samp), torch.from_numpy(data).cuda()
    else:
        npdt, mean, sd = {"u8": (np.uint8, 128, 60), "u16": (np.uint16, 40000, 9000)}[dtype]
        x = filterbank(npdt, n_chan, n_samp, 9800, mean, sd)
        xd = torch.zeros((n_chan, (n_samp + 15) // 16 * 16), dtype=getattr(torch, str(x.dtype)),
                         device="cuda")
        xd[:, :n_samp].copy_(torch.from_numpy(x))
    return freqs, ranges, n_samp, xd, oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0]


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,n_out,bin_,tile,kernel", [
    ("u8", 150, 130, 0.4, 60001, 1, 0, "pattern"), ("u8", 150, 130, 0.4, 50001, 1, 0, "sum-rows"),
    ("u4", 150, 130, 0.4, 60001, 1, 0, "pattern"), ("u16", 150, 130, 0.4, 30001, 1, 0, "pattern"),
    ("u16", 150, 130, 0.4, 30001, 1, "packed", "sum-rows"),
    ("u8", 150, 130, 0.4, 60001, 1, "packed", "pattern"),
    ("u8", 150, 130, 0.4, 30001, 2, 0, "pattern"),
])
def test_alone_ring_and_host(dtype, n_chan, n_dm, slope, n_out, bin_, tile, kernel):
    freqs, ranges, n_samp, xd, ref = _beam(dtype, n_chan, n_dm, slope, n_out, bin_)
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, dtype)
    plan.set_tile(0, tile)
    assert plan.run_kernel(0, n_out, scratch=False)[0] == kernel
    for segments in (0, 1, 8):
        got = plan.run(xd, n_samp=n_samp, segments=segments)[0].cpu().numpy()
        plan.device_status()
        np.testing.assert_array_equal(got, ref, err_msg=f"segments {segments}")
    h_in, d_out = xd.cpu().pin_memory(), plan.empty_output(n_samp)
    h_out = torch.full(d_out.shape, -1, dtype=d_out.dtype).pin_memory()
    plan.run_host(h_in, h_out, torch.zeros_like(xd), d_out, n_samp=n_samp)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(plan.split(h_out, n_samp)[0].numpy(), ref)


# The sum-row tile makes ceil(DMs / 128) x ceil(outputs / 736) units of a beam,
# the pattern tile ceil(DMs / 64) x ceil(outputs / 1472).
@pytest.mark.parametrize("dtype,n_chan,n_dm,n_out,beams,tile,sums", [
    ("u8", 100, 130, 30000, 2, "pattern", False), ("u8", 100, 130, 30000, 2, "packed", False),
    ("u4", 100, 130, 30000, 2, "pattern", False), ("u8", 600, 256, 736 * 27, 2, "pattern", True),
    ("u8", 600, 256, 1472 * 13 + 300, 2, "packed", True), ("u4", 600, 200, 736 * 11, 1, "pattern", True)])
def test_batches(dtype, n_chan, n_dm, n_out, beams, tile, sums):
    freqs, ranges, n_samp, xd, ref = _beam(dtype, n_chan, n_dm, 0.3, n_out)
    spec = ddb.BeamSpec(freqs, F_HIGH, T_SAMP, ranges, dtype, n_samp)
    runner = ddb.BatchRunner([spec] * beams, autotune=False, graph=False,
                             tiles=[[(tile, -1)]] * beams)
    dms, outs = (128, 736) if sums else (64, 1472)
    assert runner.n_items == beams * -(-n_dm // dms) * -(-n_out // outs)
    for t in runner.inputs:
        w = min(t.shape[1], xd.shape[1])
        t[:, :w].copy_(xd[:, :w])
    for _ in range(2):
        runner.run()
        runner.status()
        for i in range(beams):
            np.testing.assert_array_equal(runner.planes(i)[0].cpu().numpy(), ref)
