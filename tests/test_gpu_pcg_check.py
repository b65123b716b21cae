"""The CG residual is read every four iterations: a solve that reaches its tolerance within four products does no
more, one that needs more stops within three of the first product that reaches it."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


@pytest.mark.parametrize("solver", [stba.STBA_SOLVER_PCG_FULL, stba.STBA_SOLVER_PCG_CLUSTERS])
def test_products_past_the_tolerance(solver):
    s = scenes.make_tiny_scene(m=12, n=100, seed=12, clusters=(np.arange(12) * 3 // 12).astype(np.int32), drop=0.4)

    def products(tol, cap=500):
        with stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, s.clusters, lambda0=1e-2,
                              linear_solver=solver, pcg_tol=tol, pcg_max_iter=cap) as ctx:
            return stba.stba_lm_iteration(ctx)["linear_iterations"]

    assert products(10.0) == 4         # reached from the start
    n = products(1e-6)
    assert n % 4 == 0 and n > 4
    assert products(1e-6, cap=n - 3) == n - 3   # the cap cuts the last batch
