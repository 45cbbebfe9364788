"""Troubled-cell decisions next to their thresholds: windows built so that |D|, |xbar| or
|xbar - xhat| (Sec. 2.3.1, Steps 1-3) miss their limits by relative distances from 1e-15 to 1e-3, where
the kernel's FP32 tests must hand over to the exact chain, and data scaled by powers of two out to
where FP32 under- and overflows.  The flags must equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2304_05572_gb300 import problems as P

pytestmark = pytest.mark.gpu


def _windows(n, h, amp, seed):
    """1D density made of n blocks of 9 cells, each holding one 5-cell window at a threshold."""
    rng = np.random.default_rng(seed)
    rho = np.ones(9 * n) + amp * rng.uniform(-1, 1, 9 * n)
    for b in range(n):
        q = rho[9 * b + 2: 9 * b + 7]
        d = rng.choice([0.0, 1e-15, 1e-12, 1e-9, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3]) * rng.choice([-1, 1])
        r4 = 4 * q[0] + q[1] + q[3] - 10 * q[2]              # D = r4 + 4 q4
        rn = 2 * q[0] + q[1] - q[3]                          # N = rn - 2 q4
        kind = b % 4
        if kind == 0:
            q[4] = (rng.choice([-1, 1]) * 5 * h * (1 + d) - r4) / 4
            continue
        if kind == 1:
            c = rng.choice([-1, 1]) * 2.5 * (1 + d)
        else:
            xh = -0.5 * (q[3] - q[1]) / (q[1] + q[3] - 2 * q[2])
            c = xh + rng.choice([-1, 1]) * 0.25 * (1 + d)
        # xbar = 1.7 N / D = c
        q[4] = np.clip((1.7 * rn - c * r4) / (4 * c + 3.4), 1 - 4 * amp, 1 + 4 * amp)
    return rho


@pytest.mark.parametrize("scale", [0, 100, -100, 140, -140, 400, -400])
@pytest.mark.parametrize("zeta1", ["B", "A"])
def test_flags_at_thresholds(scale, zeta1):
    from paper_2304_05572_gb300 import _build, hgks
    _build.build()
    oracle.build()
    n = 600
    h = 1.0 / (9 * n)
    s = 2.0 ** scale
    rho = _windows(n, h, 0.05, 11) * s
    W = np.ascontiguousarray(np.stack([rho, 0.1 * rho, 2.5 * s + 0.0 * rho])[:, None, :])
    cfg = P.base_config(1, 9 * n, 1, 0.0, 1.0, bc=["extrap"] * 4, zeta1_mode=zeta1)
    Wo, dt, fo = oracle.step_flags(cfg, W)[:3]
    g = hgks.Solver(cfg)
    g.hgks_set_flag_capture(True)
    g.hgks_set_state(W)
    g.hgks_step(1e9, 1, wait=False)
    fg = g.hgks_get_flags(0, 0, 0)
    g.hgks_destroy_solver()
    want = fo[(0, 0, "normal")]
    assert np.array_equal(fg, want), int((fg != want).sum())
    if scale == 0:
        assert 0.05 < want.mean() < 0.999
