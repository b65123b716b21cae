"""The S' build at the edges of its pieces and chunks (16 pairs per piece, 64 or more per chunk, blocks stored by a
chunk that holds its whole edge and added by several otherwise) and of its camera tables (rotations at, near and
far from zero): S'_k and b_k of the first iteration against the oracle, with the rows recomputed and stored.
Bars: FP64 1e-8 per block / row, as the other S' comparisons (both sides round in FP64); mixed 1e-4: about 20
roundings of 6e-8 of the terms Jc^T Jc, of which the Schur complement of a virtual point of two observations may
leave a fiftieth."""
import numpy as np
import pytest

from oracle import camera as ocam
from oracle import stba as ostba

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import blocks, rows  # noqa: E402

ANGLES = [0.0, 1e-9, 5e-3, 0.02, 0.3]   # below, around and above the series cut of the tables (1e-2 rad)


def scene(n, seed):
    """Five cameras that all see all n points, in front of them at about 10 units."""
    rng = np.random.default_rng(seed)
    axes = rng.normal(size=(5, 3))
    w = np.array(ANGLES)[:, None] * axes / np.linalg.norm(axes, axis=1, keepdims=True)
    t = rng.normal(0, 0.3, (5, 3)) + np.array([0, 0, 10.0])
    cams = np.concatenate([w, t, rng.uniform(500, 1500, (5, 1)), rng.normal(0, 0.01, (5, 2))], 1)
    pts = rng.uniform(-1, 1, (n, 3))
    oc, op = np.tile(np.arange(5), n).astype(np.int32), np.repeat(np.arange(n), 5).astype(np.int32)
    uv = ocam.residuals(cams, pts, oc, op, np.zeros((5 * n, 2))) + rng.normal(0, 1, (5 * n, 2))
    return cams, pts, oc, op, uv


@pytest.mark.parametrize("n", [3, 15, 16, 17, 64, 65, 129])
@pytest.mark.parametrize("precision,pairs", [("fp64", 1), ("fp64", 2), ("mixed", 1), ("mixed", 2)])
def test_cluster_systems_at_piece_and_chunk_edges(n, precision, pairs):
    cams, pts, oc, op, uv = scene(n, n)
    cl = np.array([0, 1, 0, 0, 1], np.int32)
    lam = 1e-2
    step = ostba.lm_iteration(cams, pts, oc, op, uv, cl, lam, ocam.cost(cams, pts, oc, op, uv),
                              ostba.Options(lambda0=lam), keep=True)[4]["step"]
    bar = 1e-8 if precision == "fp64" else 1e-4
    with stba.stba_create(cams, pts, oc, op, uv, cl, lambda0=lam, pair_blocks=pairs,
                          precision=stba.STBA_FP64 if precision == "fp64" else stba.STBA_MIXED) as ctx:
        stba.stba_lm_iteration(ctx)
        for k in range(2):
            S, b = stba.stba_get_cluster_system(ctx, k)
            eS, eb = blocks(S, step["S_blocks"][k]), rows(b, step["b_blocks"][k], 9)
            assert eS < bar and eb < bar, (k, eS, eb)
