"""The cluster factorisation and solve at the edges of the 64-wide tiles: clusters of 1 to 5 tiles, full, one short
and one over, an odd and an even number of tile rows below a step (the update works on pairs), all in one problem
and alone, with the tensor-core steps (default) and the CUDA-core factor.  Every cluster's step against a dense
FP64 solve of the device's own S'_k.  Bar 1e-6 of each camera row: at lambda = 0.09 the scaled system has no
eigenvalue below about 0.08 and none above about 20, so the FP32 solution is within 250 x 10 x 6e-8 = 1.5e-4 of the
exact one and one FP64 refinement step squares that."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import rows  # noqa: E402

SIZES = [1, 7, 8, 14, 15, 21, 22, 28, 29, 35]   # 9, 63, 72, 126, 135, 189, 198, 252, 261, 315 unknowns


@pytest.mark.parametrize("update", [0, 1])
@pytest.mark.parametrize("sizes", [SIZES] + [[s] for s in SIZES if s > 1])
def test_cluster_steps_at_tile_edges(sizes, update):
    m = sum(sizes)
    cl = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    s = scenes.make_tiny_scene(m=m, n=30 * max(m, 4), seed=m, clusters=cl, drop=0.5 if m < 40 else 0.9)
    with stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, cl, lambda0=0.09,
                          precision=stba.STBA_MIXED, factor_update=update) as ctx:
        info = stba.stba_lm_iteration(ctx)
        assert info["failed_clusters"] == 0
        dc, _ = stba.stba_last_step(ctx)
        for k in range(len(sizes)):
            S, b = stba.stba_get_cluster_system(ctx, k)
            x = np.linalg.solve(S, b)
            e = rows(dc[cl == k].ravel(), x, 9)
            assert e < 1e-6, (k, sizes[k], e)


@pytest.mark.parametrize("m", [650, 680])
def test_solve_at_the_shared_memory_limit(m):
    """One cluster solved by two CTAs: 92 tile rows, the most whose accumulators the data-flow solve holds, and 96,
    which take the solve with cluster barriers.  Backward error below 1e-8: the FP32 solution's is about 1e-6 at
    worst (6000 unknowns, 6e-8 per rounding), and the FP64 refinement step multiplies it by the FP32 factor's own
    relative error, below 1e-2 here."""
    rng = np.random.default_rng(m)
    base = scenes.make_tiny_scene(m=m, n=200, seed=3, drop=0.97)
    n = 4 * m                                        # every point seen by 4 cameras of a window around it
    oc = np.sort((np.arange(n)[:, None] * m // n + rng.permuted(np.tile(np.arange(8), (n, 1)), axis=1)[:, :4]) % m, 1)
    op = np.repeat(np.arange(n), 4).astype(np.int32)
    oc = oc.ravel().astype(np.int32)
    pts = rng.uniform(-0.3, 0.3, (n, 3))
    from oracle import camera as ocam
    uv = ocam.residuals(base.cameras_true, pts, oc, op, np.zeros((len(oc), 2))) + rng.normal(0, 1, (len(oc), 2))
    with stba.stba_create(base.cameras, pts, oc, op, uv, np.zeros(m, np.int32), lambda0=0.09,
                          precision=stba.STBA_MIXED, solve_cluster=2) as ctx:
        info = stba.stba_lm_iteration(ctx)
        assert info["failed_clusters"] == 0
        dc, _ = stba.stba_last_step(ctx)
        S, b = stba.stba_get_cluster_system(ctx, 0)
    x = dc.ravel()
    e = np.abs(S @ x - b).max() / (np.abs(S) @ np.abs(x) + np.abs(b)).max()
    assert e < 1e-8, e


@pytest.mark.parametrize("sizes", [[1, 3, 4, 7, 8, 11, 14, 15], [3], [4], [7], [8], [300], [160, 150]])
def test_fp64_panels_at_tile_edges(sizes):
    """FP64 panels of 32 columns, a row tile per CTA or, while twice a step's tiles fit on the SMs, half a tile: clusters
    of 1 to 5 tiles around the tile edges, one of 85 tiles and two of 45 and 43, which begin with whole tiles and go
    over to halves.  Bar 1e-10 of each camera row: condition below 250 (of the system with unit diagonal, which the
    reference solves too) x 2700 roundings of 1.1e-16."""
    m = sum(sizes)
    cl = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    s = scenes.make_tiny_scene(m=m, n=max(30 * min(m, 20), 4), seed=m, clusters=cl, drop=0.5 if m < 100 else 0.9)
    with stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, cl, lambda0=0.09,
                          precision=stba.STBA_FP64) as ctx:
        info = stba.stba_lm_iteration(ctx)
        assert info["failed_clusters"] == 0
        dc, _ = stba.stba_last_step(ctx)
        for k in range(len(sizes)):
            S, b = stba.stba_get_cluster_system(ctx, k)
            d = 1 / np.sqrt(np.diag(S))
            e = rows(dc[cl == k].ravel(), d * np.linalg.solve(S * d[:, None] * d, b * d), 9)
            assert e < 1e-10, (k, sizes[k], e)
