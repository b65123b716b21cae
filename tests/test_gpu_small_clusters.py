"""Cluster solves whose CTAs mostly own no tile row or one: 400 clusters of 1 to 7 cameras (one tile of 64, one or two
of 32) solved by 2, 4 and 8 CTAs each, in several waves on the device, so that a CTA that leaves is replaced at once
by one of another cluster.  Every cluster's step against a dense FP64 solve of the device's own S'_k.  At lambda =
0.09 the scaled system of at most 63 unknowns has no eigenvalue below 0.083 (lambda / (1 + lambda)) and none above its
trace, 63: condition 760.  Bars, of each camera row: mixed precision 1e-6 (the FP32 solution is within 760 x 10 x
6e-8 = 5e-4 of the exact one and one FP64 refinement step squares that); FP64 3e-11 (760 x 63 x 1.1e-16 = 5e-12, with
a factor of five for the reference's own rounding and the rows' scales)."""
import numpy as np
import pytest

import scenes
from oracle import camera as ocam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import rows  # noqa: E402


@pytest.fixture(scope="module")
def scene():
    rng = np.random.default_rng(17)
    sizes = rng.integers(1, 8, 400)
    m = int(sizes.sum())
    base = scenes.make_tiny_scene(m=m, n=64, seed=3, drop=0.99)
    n = 6 * m                                        # every point seen by 4 cameras of a window of 8
    oc = (np.arange(n)[:, None] * m // n + rng.permuted(np.tile(np.arange(8), (n, 1)), axis=1)[:, :4]) % m
    oc = np.sort(oc, 1).ravel().astype(np.int32)
    op = np.repeat(np.arange(n), 4).astype(np.int32)
    pts = rng.uniform(-0.3, 0.3, (n, 3))
    uv = ocam.residuals(base.cameras_true, pts, oc, op, np.zeros((len(oc), 2))) + rng.normal(0, 1, (len(oc), 2))
    return base.cameras, pts, oc, op, uv, np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)


@pytest.mark.parametrize("cs", [2, 4, 8])
@pytest.mark.parametrize("precision,bar", [(stba.STBA_MIXED, 1e-6), (stba.STBA_FP64, 3e-11)])
def test_solves_of_clusters_of_one_tile(scene, precision, bar, cs):
    cams, pts, oc, op, uv, cl = scene
    with stba.stba_create(cams, pts, oc, op, uv, cl, lambda0=0.09, precision=precision, solve_cluster=cs) as ctx:
        for _ in range(3):   # the same system three times: rejected or not, the state is put back
            stba.stba_set_state(ctx, 0.09, 0.0, 0)
            stba.stba_set_params(ctx, cams, pts)
            info = stba.stba_lm_iteration(ctx)
            assert info["failed_clusters"] == 0
            dc, _ = stba.stba_last_step(ctx)
            worst = 0.0
            for k in range(cl.max() + 1):
                S, b = stba.stba_get_cluster_system(ctx, k)
                d = 1 / np.sqrt(np.diag(S))
                worst = max(worst, rows(dc[cl == k].ravel(), d * np.linalg.solve(S * d[:, None] * d, b * d), 9))
            assert worst < bar, worst
