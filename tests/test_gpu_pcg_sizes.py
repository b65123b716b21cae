"""The PCG solvers at the edges of their blocks (32 cameras per block of the vector kernels, groups of 32
observations in the camera passes, runs of several cameras per warp): the FP64 step at pcg_tol = 1e-12 against
the oracle's direct solves.  Bar: 1e-7 of each row's largest entry, the CG stopping residual amplified by the
condition of the scaled system (~1e4), as for the other CG steps."""
import numpy as np
import pytest

import scenes
from oracle import camera as ocam
from oracle import stba as ostba

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import rows  # noqa: E402


@pytest.mark.parametrize("m,n", [(3, 11), (31, 64), (32, 200), (33, 97), (65, 130)])
@pytest.mark.parametrize("solver", ["full", "split"])
def test_pcg_step_at_block_edges(m, n, solver):
    clusters = (np.arange(m) * 3 // m).astype(np.int32)
    s = scenes.make_tiny_scene(m=m, n=n, seed=m, clusters=clusters, drop=0.6)
    lam = 1e-2
    F0 = ocam.cost(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv)
    kw = dict(method="lm") if solver == "full" else {}
    _, _, _, _, rec = ostba.lm_iteration(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, s.clusters, lam, F0,
                                         ostba.Options(lambda0=lam), **kw)
    which = stba.STBA_SOLVER_PCG_FULL if solver == "full" else stba.STBA_SOLVER_PCG_CLUSTERS
    with stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, s.clusters, lambda0=lam,
                          linear_solver=which, pcg_tol=1e-12, pcg_max_iter=2000) as ctx:
        info = stba.stba_lm_iteration(ctx)
        dc, dp = stba.stba_last_step(ctx)
    assert rows(dc, rec["dc"], 9) < 1e-7, rows(dc, rec["dc"], 9)
    assert rows(dp, rec["dp"], 3) < 1e-7, rows(dp, rec["dp"], 3)
    assert info["accepted"] == rec["accepted"]
