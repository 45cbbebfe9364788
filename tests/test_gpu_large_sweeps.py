"""The kernels of large sweeps (49152 interface segments and more) where the parity tests' grids take the
small sweeps' kernels: WENO-AO everywhere on the compacted passes with one item per lane, 1D grids, the
Prandtl fix, grids with one large and one small sweep.  Steps as in test_gpu_parity.check_step: identical dt
and first-stage flags, state within 1e-11; the timing classes show which form ran.  Batches of such solvers
equal their solo runs bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2304_05572_gb300 import hgks, problems as P
from test_gpu_parity import check_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2304_05572_gb300 import _build
    _build.build()
    oracle.build()


def _case(name):
    if name == "wenoao_231x230":                  # every side and pass troubled: above 32768 items a pass
        cfg, W, _ = P.random_smooth_2d(231, 230)
        return dict(cfg, recon_mode="wenoao"), W
    if name == "linear_231x230":
        cfg, W, _ = P.random_smooth_2d(231, 230)
        return dict(cfg, recon_mode="linear"), W
    if name == "hybrid_231x230":                  # few troubled items: lane groups
        return P.riemann4_2d(231, ny=230)[:2]
    if name == "tube_320x160_pr073":
        return P.viscous_shock_tube(320, 160, Re=1000.0, prandtl=0.73)[:2]
    if name == "x_small_y_large_8000x6":          # 48006 and 56000 segments
        return P.random_smooth_2d(8000, 6)[:2]
    if name == "x_large_y_small_6x8000":
        return P.random_smooth_2d(6, 8000)[:2]
    cfg, W, _ = P.sod_1d(50000)
    if name == "sod_50000_wenoao":
        cfg = dict(cfg, recon_mode="wenoao")
    if name == "sod_50000_pr073":
        cfg = dict(cfg, viscous=1, mu=1e-5, prandtl=0.73)
    return cfg, W


CASES = ["wenoao_231x230", "linear_231x230", "hybrid_231x230", "tube_320x160_pr073", "x_small_y_large_8000x6",
         "x_large_y_small_6x8000", "sod_50000", "sod_50000_wenoao", "sod_50000_pr073"]


@pytest.mark.parametrize("name", CASES)
def test_steps_match_the_oracle(name):
    cfg, W = _case(name)
    Wo = check_step(cfg, W, name)[0]
    check_step(cfg, Wo, name + ", second step")
    s = hgks.Solver(cfg)
    s.hgks_set_state(np.ascontiguousarray(W))
    s.hgks_set_timing(True)
    s.hgks_step(1e9, 1)
    calls = {k: v[1] for k, v in s.hgks_get_timing().items()}
    s.hgks_destroy_solver()
    # launches of the compacted passes: only the large sweeps' form has any
    assert calls["raw_normal_flags"] == 2 and calls["normal_weno_ao"] == 2
    assert calls["tangential_weno_ao"] == (2 if cfg["dim"] == 2 else 0)
    mixed = name.startswith("x_")
    assert calls["gks_flux"] == (4 if mixed else 2)


def _batch_equals_alone(cases, steps, **kw):
    import torch
    stream = torch.cuda.Stream()
    solvers = []
    for cfg, W in cases:
        s = hgks.Solver(cfg, stream=stream)
        s.hgks_set_state(np.ascontiguousarray(W))
        solvers.append(s)
    b = hgks.Batch(solvers, stream=stream)
    b.hgks_batch_step([1e9] * len(cases), nsteps=steps, **kw)
    assert b.hgks_batch_sync() == (len(cases), 0)
    for k, ((cfg, W), s) in enumerate(zip(cases, solvers)):
        a = hgks.Solver(cfg)
        a.hgks_set_state(np.ascontiguousarray(W))
        assert a.hgks_step(1e9, steps) == steps
        assert np.array_equal(s.hgks_get_state(), a.hgks_get_state()), k
        assert s.hgks_get_time() == a.hgks_get_time()
        a.hgks_destroy_solver()
    b.hgks_batch_destroy()
    for s in solvers:
        s.hgks_destroy_solver()


@pytest.mark.parametrize("graph,autotune", [(False, False), (True, True)])
def test_batch_2d_bitwise_equal_to_alone(graph, autotune):
    cases = [_case(n) for n in CASES if not n.startswith("sod")]
    cases += [P.riemann4_2d(37, ny=29)[:2], P.viscous_shock_tube(48, 24, Re=1000.0, prandtl=0.73)[:2]]
    _batch_equals_alone(cases, 6, graph=graph, autotune=autotune)


@pytest.mark.parametrize("graph,autotune", [(False, False), (True, True)])
def test_batch_1d_bitwise_equal_to_alone(graph, autotune):
    cases = [P.sod_1d(200)[:2]] + [_case(n) for n in CASES if n.startswith("sod")]
    _batch_equals_alone(cases, 6, graph=graph, autotune=autotune)
