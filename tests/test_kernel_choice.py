"""Which kernel a launch takes (dd_plan_run_kernel), on the host: the sum-row and
direct tiles where their rules say so, and the tiles they replace elsewhere."""
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import _lib
from synth import channel_freqs


def _plan(dtype, n_chan, n_dm, slope, bin_=1, f_high=1500.0, band=300.0, t_samp=64e-6):
    freqs = channel_freqs(f_high, band, n_chan)
    step = slope * bin_ * t_samp / oracle.delay_coeff(freqs[-1], f_high)
    return dd.Plan(freqs, f_high, t_samp, [(0.0, n_dm * step, step, bin_)], dtype, upload=False)


# dtype, channels, DMs, slope, bin -> with scratch, without
SUM_ROWS = [
    ("u8", 600, 200, 0.2, 1, ("sum-rows", True), ("sum-rows", False)),
    ("u4", 700, 200, 0.2, 1, ("sum-rows", True), ("sum-rows", False)),
    ("u16", 600, 200, 0.2, 1, ("sum-rows", False), ("sum-rows", False)),
    ("u8", 4099, 128, 2.5, 1, ("sum-rows", False), ("sum-rows", False)),  # its copy's window is too wide
    ("u8", 500, 1024, 0.2, 2, ("sum-rows", False), ("sum-rows", False)),
    ("u8", 500, 1024, 0.2, 4, ("pattern", False), ("pattern", False)),
    ("u8", 95, 200, 0.2, 1, ("pattern", True), ("pattern", False)),
    ("u8", 128, 1024, 1.0, 1, ("pattern", True), ("pattern", False)),  # few channels share a row
    ("f32", 600, 200, 0.2, 1, ("pattern", False), ("pattern", False)),
]


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,bin_,with_scratch,without", SUM_ROWS)
def test_sum_row_tile_choice(dtype, n_chan, n_dm, slope, bin_, with_scratch, without):
    plan = _plan(dtype, n_chan, n_dm, slope, bin_)
    assert plan.run_kernel(0, 20000, scratch=True) == with_scratch
    assert plan.run_kernel(0, 20000, scratch=False) == without
    if without[0] == "sum-rows":  # an explicit shape keeps the pattern kernel
        plan.set_tile_shape(0, "pattern", 0)
        assert plan.run_kernel(0, 20000) == ("pattern", False)


def test_packed_tile_choice():
    for dtype, n_chan, slope, bin_, want in (("u8", 600, 0.2, 1, "sum-rows"),
                                             ("u8", 4099, 2.5, 1, "sum-rows"),
                                             ("u8", 600, 0.2, 8, "sum-rows"),
                                             ("u8", 95, 0.2, 1, "pattern")):
        plan = _plan(dtype, n_chan, 128, slope, bin_)
        plan.set_tile(0, "packed")
        for scratch in (True, False):
            assert plan.run_kernel(0, 2000, scratch) == (want, True)


def test_direct_tile_choice():
    """Steep plans: the direct tile for long launches, the offset tile for short."""
    for dtype in ("u8", "u16", "f32"):
        plan = _plan(dtype, 64, 256, 8.0, 1, 400.0, 100.0, 327.68e-6)
        assert plan.run_kernel(0, 1 << 20)[0] == "direct"
        assert plan.run_kernel(0, 1000)[0] == "offset"
        plan.set_tile(0, 2)
        assert plan.run_kernel(0, 1 << 20)[0] == "offset"


def test_run_kernel_arguments():
    plan = _plan("u8", 64, 64, 0.2)
    for args, status in (((1, 100), _lib.DD_ERR_INVALID_ARG), ((-1, 100), _lib.DD_ERR_INVALID_ARG),
                         ((0, 0), _lib.DD_ERR_SHAPE)):
        with pytest.raises(dd.DDError) as err:
            plan.run_kernel(*args)
        assert err.value.status == status


@pytest.mark.parametrize("dtype,n_dm,n_out,want", [
    # whole waves of 152 CTAs: 45 x 4 direct (2 waves) against 26 x 17 offset (3)
    ("f32", 400, 16384, "offset"), ("u16", 400, 16384, "offset"), ("u8", 400, 32768, "offset"),
    ("f32", 200, 32000, "offset"),
    # 42 x 3 (1 wave) against 24 x 15 (3); 82 x 3 (2) against 47 x 15 (5)
    ("f32", 356, 15360, "direct"), ("f32", 356, 30001, "direct"), ("u8", 356, 60002, "direct"),
])
def test_direct_tile_takes_whole_waves_into_account(dtype, n_dm, n_out, want):
    plan = _plan(dtype, 336, n_dm, 5.5, 1, 400.0, 100.0, 327.68e-6)
    assert plan.info(0)["tile_dms"] == [2]
    assert plan.run_kernel(0, n_out)[0] == want


@pytest.mark.parametrize("dtype,n_chan,n_dm,slope,bin_,n_out,want", [
    # 2 x 82 units of 128 DMs (2 waves of 152) against 3 x 41 of 64 (1)
    ("u8", 150, 130, 0.4, 1, 60000, "pattern"), ("u8", 300, 130, 1.0, 1, 60000, "pattern"),
    ("u4", 150, 130, 0.4, 1, 60000, "pattern"), ("u16", 150, 130, 0.4, 1, 30000, "pattern"),
    ("u8", 150, 130, 0.4, 1, 50000, "sum-rows"), ("u8", 1500, 130, 0.4, 1, 60000, "sum-rows"),
    ("u8", 150, 512, 0.4, 1, 73600, "sum-rows"), ("u16", 150, 130, 0.4, 1, 20000, "sum-rows"),
    ("u8", 150, 130, 0.4, 2, 30000, "pattern"), ("u8", 700, 1000, 0.4, 2, 66240, "sum-rows"),
])
def test_sum_row_tile_takes_whole_waves_into_account(dtype, n_chan, n_dm, slope, bin_, n_out, want):
    plan = _plan(dtype, n_chan, n_dm, slope, bin_)
    assert plan.run_kernel(0, n_out, scratch=False) == (want, False)


def test_packed_uint16_never_reads_the_input_with_its_copys_tables():
    """DD_TILE_PACKED uint16 has pattern tables for its copy alone: from the input
    it stays on the sum-row tile where the rule would prefer the pattern tile."""
    plan = _plan("u16", 150, 130, 0.4)
    plan.set_tile(0, "packed")
    assert plan.run_kernel(0, 30000) == ("sum-rows", False)


def test_choice_over_many_waves():
    """Past 64 waves the mean of the units decides, as it nearly does just below."""
    plan = _plan("u8", 600, 1000, 0.2)
    per_wave = 152 * 736 // 8  # 8 blocks of 128 DMs
    for waves in (50, 63, 64, 65, 2000):
        assert plan.run_kernel(0, waves * per_wave, scratch=False)[0] == "sum-rows"
