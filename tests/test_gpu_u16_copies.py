"""Packed copies of uint16 input on a plan whose range runs on the sum-row tile
from the input: the calls that take copies or scratch for them still do what
they document."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import _lib
from synth import channel_freqs, filterbank

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

F_HIGH, T_SAMP, N_CHAN, N_DM, N_SAMP = 1500.0, 64e-6, 600, 200, 9001


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def beam():
    freqs = channel_freqs(F_HIGH, 300.0, N_CHAN)
    step = 0.2 * T_SAMP / oracle.delay_coeff(freqs[-1], F_HIGH)
    ranges = [(0.0, N_DM * step, step, 1)]
    x = filterbank(np.uint16, N_CHAN, N_SAMP, 9400, 40000, 9000)
    xd = torch.zeros((N_CHAN, (N_SAMP + 7) // 8 * 8), dtype=torch.uint16, device="cuda")
    xd[:, :N_SAMP].copy_(torch.from_numpy(x).cuda())
    return freqs, ranges, xd, oracle.forward(x, freqs, F_HIGH, T_SAMP, ranges)[0]


def _stream():
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("tile", [0, "packed"])
def test_run_packed_reads_the_copies(beam, tile):
    """dd_run_packed works on the copies dd_pack_input made: the input's memory
    may have been given another use by then."""
    freqs, ranges, xd, ref = beam
    lib = _lib.load()
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, "u16")
    plan.set_tile(0, tile)
    n = plan.packed_scratch_bytes(N_SAMP, 1)
    scratch = torch.zeros(n, dtype=torch.uint8, device="cuda")
    x = xd.clone()
    out = plan.empty_output(N_SAMP)
    _lib.check(lib.dd_pack_input(plan.handle, x.data_ptr(), x.stride(0), N_SAMP,
                                 scratch.data_ptr(), n, _stream()))
    x.zero_()
    _lib.check(lib.dd_run_packed(plan.handle, x.data_ptr(), x.stride(0), N_SAMP, out.data_ptr(),
                                 scratch.data_ptr(), n, _stream()))
    plan.device_status()
    np.testing.assert_array_equal(plan.split(out, N_SAMP)[0].cpu().numpy(), ref)


@pytest.mark.parametrize("tile", [0, "packed"])
@pytest.mark.parametrize("segments", [8, 3, 1])
def test_run_takes_the_scratch_the_query_names(beam, tile, segments):
    """dd_run_scratch with exactly the ring (or the full copies) that
    dd_plan_packed_scratch_bytes gives for the segments."""
    freqs, ranges, xd, ref = beam
    lib = _lib.load()
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, "u16")
    plan.set_tile(0, tile)
    n = plan.packed_scratch_bytes(N_SAMP, segments)
    assert 0 < n and (segments < 8 or n < plan.packed_scratch_bytes(N_SAMP, 1))
    scratch = torch.zeros(n, dtype=torch.uint8, device="cuda")
    out = plan.empty_output(N_SAMP)
    _lib.check(lib.dd_run_scratch(plan.handle, xd.data_ptr(), xd.stride(0), N_SAMP, out.data_ptr(),
                                  scratch.data_ptr(), n, _stream()))
    plan.device_status()
    np.testing.assert_array_equal(plan.split(out, N_SAMP)[0].cpu().numpy(), ref)


def test_packed_tile_still_refuses_missing_and_short_scratch(beam):
    freqs, ranges, xd, _ = beam
    lib = _lib.load()
    plan = dd.Plan(freqs, F_HIGH, T_SAMP, ranges, "u16")
    plan.set_tile(0, "packed")
    out = plan.empty_output(N_SAMP)
    scratch = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    for ptr, n, status in ((None, 0, _lib.DD_ERR_UNSUPPORTED),
                           (scratch.data_ptr(), 4096, _lib.DD_ERR_BUDGET)):
        assert lib.dd_run_scratch(plan.handle, xd.data_ptr(), xd.stride(0), N_SAMP,
                                  out.data_ptr(), ptr, n, _stream()) == status
    keep = (ctypes.c_int64 * 1)(100)
    ring = plan.packed_scratch_bytes(N_SAMP, 8)
    scratch = torch.zeros(ring, dtype=torch.uint8, device="cuda")
    assert lib.dd_run_window(plan.handle, xd.data_ptr(), xd.stride(0), N_SAMP, keep,
                             out.data_ptr(), scratch.data_ptr(), ring,
                             _stream()) == _lib.DD_ERR_BUDGET
