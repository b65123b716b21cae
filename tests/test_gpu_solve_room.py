"""One cluster solved by two CTAs on both sides of the largest system whose accumulators fit in a CTA's shared memory
(the data-flow solve) and of the switch to the solve with cluster barriers, found from the device's limit: FP32 factor
(tiles of 64) and FP64 (tiles of 32).  Backward error of the step for the device's own S' and b', below 1e-8 with the
FP32 factor (about 1e-6 at worst from 6000 unknowns x 6e-8, times the FP32 factor's own relative error, below 1e-2,
by the refinement step) and 1e-12 in FP64 (3000 unknowns x 1.1e-16 x 3)."""
import numpy as np
import pytest

import scenes
from oracle import camera as ocam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


def push_bytes(nt, tile, real, cs=2):
    """shared memory of a data-flow solve's CTA: barriers, the vector, and per owned tile row its right-hand side and the
    256 threads' 16-byte sums, nine scratch rows"""
    slots = -(-nt // cs)
    return 16 * nt + real * (nt * tile + slots * (tile + 256 * (16 // real)) + 9 * tile) + 16


def largest(tile, real):
    room = torch.cuda.get_device_properties(0).shared_memory_per_block_optin
    return max(nt for nt in range(1, 1000) if push_bytes(nt, tile, real) <= room)


@pytest.mark.parametrize("past", [0, 1])
@pytest.mark.parametrize("precision,tile,real,bar", [(stba.STBA_MIXED, 64, 4, 1e-8), (stba.STBA_FP64, 32, 8, 1e-12)])
def test_solve_on_both_sides_of_the_limit(precision, tile, real, bar, past):
    nt = largest(tile, real) + past
    m = nt * tile // 9                       # the last tile row is partly padding
    assert -(-9 * m // tile) == nt
    rng = np.random.default_rng(m)
    base = scenes.make_tiny_scene(m=m, n=200, seed=3, drop=0.97)
    n = 4 * m                                # every point seen by 4 cameras of a window around it
    oc = (np.arange(n)[:, None] * m // n + rng.permuted(np.tile(np.arange(8), (n, 1)), axis=1)[:, :4]) % m
    oc = np.sort(oc, 1).ravel().astype(np.int32)
    op = np.repeat(np.arange(n), 4).astype(np.int32)
    pts = rng.uniform(-0.3, 0.3, (n, 3))
    uv = ocam.residuals(base.cameras_true, pts, oc, op, np.zeros((len(oc), 2))) + rng.normal(0, 1, (len(oc), 2))
    with stba.stba_create(base.cameras, pts, oc, op, uv, np.zeros(m, np.int32), lambda0=0.09, precision=precision,
                          solve_cluster=2) as ctx:
        info = stba.stba_lm_iteration(ctx)
        assert info["failed_clusters"] == 0
        dc, _ = stba.stba_last_step(ctx)
        S, b = stba.stba_get_cluster_system(ctx, 0)
    x = dc.ravel()
    e = np.abs(S @ x - b).max() / (np.abs(S) @ np.abs(x) + np.abs(b)).max()
    assert e < bar, (m, e)
