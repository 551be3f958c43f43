"""Scratch that Plan.run takes for packed copies: none where no range reads one."""
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from synth import channel_freqs


def _plan(dtype, n_chan):
    freqs = channel_freqs(1500.0, 300.0, n_chan)
    step = 0.2 * 64e-6 / oracle.delay_coeff(freqs[-1], 1500.0)
    return dd.Plan(freqs, 1500.0, 64e-6, [(0.0, 200 * step, step, 1)], dtype, upload=False)


def test_uint16_on_the_sum_row_tile_takes_none():
    pytest.importorskip("torch")
    n = 20000
    plan = _plan("u16", 600)
    assert plan.info(n)["packed_copy"] == [True] and plan.run_kernel(0, 19000) == ("sum-rows", False)
    for segments in (8, 1, 0):
        assert plan._input_scratch(n, "cpu", segments) is None
    plan.set_tile(0, "packed")  # asked for: the call still needs it
    assert plan._input_scratch(n, "cpu", 8).numel() == plan.input_scratch_bytes(n) > 0


def test_other_plans_take_theirs():
    pytest.importorskip("torch")
    n = 20000
    for dtype, n_chan in (("u16", 64), ("u8", 600), ("u4", 600), ("u8", 64)):
        plan = _plan(dtype, n_chan)
        assert plan._input_scratch(n, "cpu", 8).numel() == plan.packed_scratch_bytes(n, 8) > 0
        assert plan._input_scratch(n, "cpu", 1).numel() == plan.packed_scratch_bytes(n, 1) > 0
