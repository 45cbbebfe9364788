"""GPU steps against the oracle where the flux's exponential and erfc leave their usual range:
|sqrt(lambda) U| around and beyond 8 (the library erfc takes over there), dt/(2 tau) from nearly 0 to far
beyond the exponential's range, and tau = 0 reached through c1 = 0 on equal pressures.  Bounds as for
every other step of the parity tests: 1e-11 of the component's scale."""
import numpy as np
import pytest

import oracle
from paper_2304_05572_gb300 import problems as P

pytestmark = pytest.mark.gpu


def _waves(dim, nx, ny, u, v, p0, amp):
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    s = np.sin(2 * np.pi * x)[None, :] * np.ones(ny)[:, None]
    c = np.cos(2 * np.pi * y)[:, None] * np.ones(nx)[None, :] if dim == 2 else 0.0 * s
    return P.conservative(1.0 + amp * s, u * (1 + amp * c), v * (1 - amp * s), p0 * (1 + amp * (s + c)), dim=dim)


CASES = {
    # U / sqrt(2 h) = 7.9 and 8.1 (both sides of the switch within the wave), and far beyond
    "mach_edge": dict(u=8.0 * np.sqrt(2.0), p0=1.0, amp=0.02),
    "mach_20": dict(u=-24.0, p0=1.0, amp=0.02),
    # c1 = 0: tau = c2 |dp| / sum p dt, tiny where the pressure is nearly flat
    "stiff_tau": dict(u=0.3, p0=1.0, amp=1e-4, c1=0.0),
    "zero_tau_flat_pressure": dict(u=0.3, p0=1.0, amp=0.0, c1=0.0),
    # tau >> dt: the exponent is nearly 0
    "soft_tau": dict(u=0.3, p0=1.0, amp=0.1, viscous=1, mu=20.0, c1=0.0, fixed_dt=1e-4),
}


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_step_matches_oracle(name, dim):
    from paper_2304_05572_gb300 import _build, hgks
    _build.build()
    oracle.build()
    k = dict(CASES[name])
    nx, ny = (75, 1) if dim == 1 else (33, 18)
    W = np.ascontiguousarray(_waves(dim, nx, ny, k.pop("u"), 0.4 if dim == 2 else 0.0, k.pop("p0"), k.pop("amp"))).reshape(dim + 2, ny, nx)
    cfg = P.base_config(dim, nx, ny, 0.0, 1.0, 0.0, 1.0, **k)
    s = hgks.Solver(cfg)
    s.hgks_set_state(W)
    assert s.hgks_step(1e9, 1) == 1
    Wg = s.hgks_get_state()
    s.hgks_destroy_solver()
    Wo, _, n, _ = oracle.run(cfg, W, 1e9, max_steps=1)
    assert n == 1
    scale = np.abs(Wo).reshape(dim + 2, -1).max(1)
    scale = np.maximum(scale, 1e-3 * scale.max())
    err = (np.abs(Wg - Wo).reshape(dim + 2, -1).max(1) / scale).max()
    assert err <= 1e-11, err
