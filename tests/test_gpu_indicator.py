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


@pytest.mark.parametrize("nx,ny", [(7101, 7), (12300, 4), (9900, 5), (231, 230)])
def test_large_sweep_tangential_flags_ragged(nx, ny):
    """Sweeps from 49152 segments on: the flag kernel takes 4 lines and one pass per thread, 32 interfaces
    per warp; sides that leave 1, 2, 3 and 0 lines in the last group and interfaces across the group edge.
    First-stage flags are decided on identical inputs, so they and the counters are exact."""
    from paper_2304_05572_gb300 import _build, hgks
    _build.build()
    oracle.build()
    cfg, W, _ = P.riemann4_2d(nx, ny=ny)
    fo = oracle.step_flags(cfg, W)[2]
    g = hgks.Solver(cfg)
    g.hgks_set_flag_capture(True)
    g.hgks_set_state(W)
    g.hgks_step(1e9, 1, wait=False)
    st = g.hgks_get_stats()
    for d in range(2):
        fg = g.hgks_get_flags(0, d, 1)
        assert np.array_equal(fg, fo[(0, d, "tang")]), d
        assert fg.any()
        assert st["troubled"][0, d, 1] == sum(bin(v).count("1") * int((fg == v).sum()) for v in range(16))
        assert st["examined"][0, d, 1] == 4 * fg.size
    g.hgks_destroy_solver()
