"""The range-checked build (HGKS_DEBUG_BOUNDS) on the kernels of large sweeps, which
test_gpu_debug_build's grids do not reach: ragged 2D, WENO-AO everywhere, one large and one small
sweep, 1D, and a batch of them.  No access leaves the solver's buffers, and one step agrees with the normal
build's within twice the per-step parity bound (each build is within 1e-11 of the oracle; their free-order
parts may fuse products differently)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = r'''
import sys
import numpy as np
out_path, root = sys.argv[1:]
sys.path.insert(0, root)
from paper_2304_05572_gb300 import hgks, problems as P
smooth, strip, sod = P.random_smooth_2d(231, 230), P.random_smooth_2d(8000, 6), P.sod_1d(50001)
cases = {"riemann": P.riemann4_2d(333, ny=229)[:2], "smooth_wenoao": (dict(smooth[0], recon_mode="wenoao"), smooth[1]),
         "tube": P.viscous_shock_tube(320, 160, Re=1000.0, prandtl=0.73)[:2], "strip": strip[:2], "sod": sod[:2],
         "sod_wenoao": (dict(sod[0], recon_mode="wenoao", viscous=1, mu=1e-5, prandtl=0.73), sod[1])}
out = {}
for name, (cfg, W) in cases.items():
    out[name] = hgks.run(cfg, W, 1e9, max_steps=1)[0]
for dim in (1, 2):
    sv = []
    for cfg, W in cases.values():
        if cfg["dim"] == dim:
            sv.append(hgks.Solver(cfg))
            sv[-1].hgks_set_state(np.ascontiguousarray(W))
    b = hgks.Batch(sv)
    b.hgks_batch_step([1e9] * len(sv), nsteps=1, graph=False)
    b.hgks_batch_sync()
    for k, s in enumerate(sv):
        out["batch%d_%d" % (dim, k)] = s.hgks_get_state()
    b.hgks_batch_destroy()
np.savez(out_path, bounds=np.array(hgks.hgks_debug_bounds()[:2], dtype=np.int64), **out)
'''


def _run(debug, path):
    env = dict(os.environ)
    env.pop("HGKS_DEBUG_BOUNDS", None)
    if debug:
        env["HGKS_DEBUG_BOUNDS"] = "1"
    r = subprocess.run([sys.executable, "-c", RUN, str(path), ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return np.load(path)


def test_no_out_of_range_access(tmp_path):
    from paper_2304_05572_gb300 import _build
    _build.build()
    _build.build(debug=True)
    dbg, ref = _run(True, tmp_path / "d.npz"), _run(False, tmp_path / "r.npz")
    assert dbg["bounds"].tolist() == [1, 0] and ref["bounds"].tolist() == [0, 0]
    for key in ref.files:
        if key != "bounds":
            a, b = dbg[key], ref[key]
            assert np.max(np.abs(a - b)) <= 2e-11 * np.max(np.abs(b)), key
