"""The benchmark's roofline counts what runs on the FP64 pipe: at the times measured on one GB300 (1024^2
four-quadrant step, 152 SMs at 2070 MHz) the fractions stay below 1 and agree with the profiler's utilisation of
that pipe (88 % of the flux launches, counters divided by the same issue rate) within the profiler's own spread."""
import pytest

import bench


def test_fractions_at_the_measured_times():
    achieved, peak, frac = bench.flux_roofline(1024, 3.49, 152, 2070.0)
    assert peak == pytest.approx(152 * 4 * 32 / 64 * 2070e6)
    assert frac == achieved / peak and 0.86 < frac < 0.92
    achieved, peak, frac = bench.step_roofline(237.8, 152, 2070.0)
    assert frac == achieved / peak and 0.75 < frac < 0.9
    # the flux launches are part of the step
    assert 4 * 1025 / 1024 * bench.FLUX_FP64_INSTR_PER_GP < bench.STEP_FP64_INSTR_PER_CELL_STAGE


def test_small_sweeps_have_no_flux_roofline():
    assert bench.flux_roofline(221, 1.0, 152, 2070.0) is None
    assert bench.flux_roofline(222, 1.0, 152, 2070.0) is not None
