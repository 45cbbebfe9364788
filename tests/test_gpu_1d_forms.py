"""1D sweeps on both sides of the sizes where they leave the small sweeps' lane groups for the compacted
passes: hybrid and WENO-AO everywhere from 32768 reconstructed sides on (16383 cells), linear from 49152
interfaces (49151 cells): steps against the oracle (test_gpu_parity.check_step), the form by the timing
classes, and a batch of both forms and the allocation-free step (whose scratch holds what earlier calls left)
against solo runs."""
import numpy as np
import pytest

import oracle
from paper_2304_05572_gb300 import hgks, problems as P
from test_gpu_large_sweeps import _batch_equals_alone
from test_gpu_parity import check_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2304_05572_gb300 import _build
    _build.build()
    oracle.build()


def _case(n, mode="wenoao", **kw):
    cfg, W, _ = P.sod_1d(n)
    return dict(cfg, recon_mode=mode, **kw), W


@pytest.mark.parametrize("n,mode,compacted", [(16382, "wenoao", False), (16383, "wenoao", True), (20000, "wenoao", True),
                                              (16382, "hybrid", False), (16383, "hybrid", True),
                                              (49150, "linear", False), (49151, "linear", True)])
def test_form_and_parity(n, mode, compacted):
    cfg, W = _case(n, mode)
    check_step(cfg, W, "%s sod %d" % (mode, n))
    s = hgks.Solver(cfg)
    s.hgks_set_state(np.ascontiguousarray(W))
    s.hgks_set_timing(True)
    s.hgks_step(1e9, 1)
    assert s.hgks_get_timing()["normal_weno_ao"][1] == (2 if compacted else 0)
    s.hgks_destroy_solver()


@pytest.mark.parametrize("graph,autotune", [(False, False), (True, True)])
def test_batch_of_both_forms(graph, autotune):
    cases = [_case(16382), _case(16383), _case(16382, "hybrid"), _case(16383, "hybrid"),
             _case(20000, "linear"), _case(16500, viscous=1, mu=1e-5, prandtl=0.73)]
    _batch_equals_alone(cases, 6, graph=graph, autotune=autotune)


def test_allocation_free_step():
    import torch
    for n, mode in ((37105, "hybrid"), (16382, "wenoao"), (16383, "wenoao"), (37105, "linear")):
        cfg, W = _case(n, mode)
        a = hgks.Solver(cfg)
        a.hgks_set_state(np.ascontiguousarray(W))
        assert a.hgks_step(1e300, 1) == 1
        d = torch.from_numpy(np.ascontiguousarray(W)).cuda()
        out, status = torch.empty_like(d), torch.full((1,), -9, dtype=torch.int32, device="cuda")
        hgks.hgks_step_noalloc(cfg, d, out, status=status)
        torch.cuda.synchronize()
        assert status.item() == 0 and np.array_equal(out.cpu().numpy(), a.hgks_get_state()), (n, mode)
        a.hgks_destroy_solver()
