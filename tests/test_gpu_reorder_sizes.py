"""A new assignment's virtual points and camera lists at the edges of their blocks: 256 observations of a camera per
row, 2048 per chunk, 2048 observations per scan tile and 64 tiles per sum; cameras of more than 16384 observations,
whose lists come from the scan over all observations instead.  Two assignments in turn, cameras with and without
companions in their cluster; the FP64 step after each against the oracle's, 1e-7 of each row's largest entry (atomic
sums through the condition of the damped system), and the exact counts."""
import numpy as np
import pytest

import scenes
from oracle import camera as ocam
from oracle import stba as ostba

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import rows  # noqa: E402


@pytest.mark.parametrize("m,n", [(4, 15), (5, 255), (5, 257), (4, 2047), (4, 2048), (4, 2049), (3, 4097), (24, 6000),
                                 (4, 16384), (4, 16385)])
def test_reordering_at_block_edges(m, n):
    first = np.r_[0, 0, 1, np.full(m - 3, 1)].astype(np.int32)    # camera 2 (and the rest) and cameras 0, 1
    second = np.r_[0, 1, 0, np.full(m - 3, 2)].astype(np.int32) if m > 3 else np.array([0, 1, 0], np.int32)
    s = scenes.make_tiny_scene(m=m, n=n, seed=m + n, clusters=first, drop=0.0)
    keep = np.ones(len(s.obs_cam), bool)
    keep[(s.obs_cam == 1) & (s.obs_pt % 3 == 0)] = False           # camera 0 alone on every third point
    oc, op, uv = s.obs_cam[keep], s.obs_pt[keep], s.obs_uv[keep]
    lam = 1e-2
    with stba.stba_create(s.cameras, s.points, oc, op, uv, first, lambda0=lam, precision=stba.STBA_FP64) as ctx:
        for cl in (first, second):
            stba.stba_set_clusters(ctx, cl)
            c0, p0 = (np.array(x) for x in stba.stba_get_params(ctx))
            lam, F = stba.stba_get_state(ctx)[0], ocam.cost(c0.reshape(m, 9), p0.reshape(n, 3), oc, op, uv)
            rec = ostba.lm_iteration(c0.reshape(m, 9), p0.reshape(n, 3), oc, op, uv, cl, lam, F,
                                     ostba.Options(lambda0=lam))[4]
            stba.stba_lm_iteration(ctx)
            dc, dp = stba.stba_last_step(ctx)
            key = op.astype(np.int64) * m + cl[oc]
            sizes = np.unique(key, return_counts=True)[1].astype(np.int64)
            info = stba.stba_problem_info(ctx)
            assert info["nv"] == len(sizes) and info["pair_instances"] == np.sum(sizes * (sizes - 1) // 2)
            assert rows(dc, rec["dc"], 9) < 1e-7, rows(dc, rec["dc"], 9)
            assert rows(dp, rec["dp"], 3) < 1e-7, rows(dp, rec["dp"], 3)
