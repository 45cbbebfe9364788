"""Troubled-cell decisions where Step 1's limit and the data lie at the lower end of FP32: cells so small that
Z1 = 5 h (reading B) is 1.5 times the smallest normal float or a little above, with data of the same size,
whose FP32 image is zero.  The flags must equal the oracle's bit for bit.  Scaling the domain and the data
alike leaves every decision as it is, so the flags also equal those of the unscaled problem."""
import numpy as np
import pytest

import oracle
from paper_2304_05572_gb300 import problems as P

pytestmark = pytest.mark.gpu


def _flags(scale, n):
    from paper_2304_05572_gb300 import hgks
    s = 2.0 ** scale
    rng = np.random.default_rng(3)
    rho = s * rng.uniform(0.3, 0.95, n)
    W = np.ascontiguousarray(np.stack([rho, 0.1 * rho, 2.5 * s + 0.0 * rho])[:, None, :])
    cfg = P.base_config(1, n, 1, 0.0, n * 0.3 * s, bc=["extrap"] * 4, cfl=0.1, c1=0.05)   # Z1 = 1.5 s
    want = oracle.step_flags(cfg, W)[2][(0, 0, "normal")]
    g = hgks.Solver(cfg)
    g.hgks_set_flag_capture(True)
    g.hgks_set_state(W)
    g.hgks_step(1e9, 1, wait=False)
    got = g.hgks_get_flags(0, 0, 0)
    g.hgks_destroy_solver()
    return got, want


@pytest.mark.parametrize("n", [2000, 60000])      # the small and the large sweeps' flag kernels
@pytest.mark.parametrize("scale", [-126, -122, -110])
def test_flags_at_the_lower_end_of_fp32(scale, n):
    from paper_2304_05572_gb300 import _build
    _build.build()
    oracle.build()
    got, want = _flags(scale, n)
    assert 0.05 < want.mean() < 0.999
    assert np.array_equal(got, want), int((got != want).sum())
    assert np.array_equal(want, _flags(0, n)[1])
