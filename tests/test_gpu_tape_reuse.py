"""A tape restarted in the buffers that it has (as long or shorter), in longer ones and after being freed gives the
gradients of a fresh context's and holds exactly the iterations asked for.  FP64; the bar, 1e-8 of the largest entry,
allows for the order of the atomic sums (1e-16 each) through a step's condition (~1e4 a step, three steps)."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


def _ctx(s):
    return stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, s.clusters, lambda0=0.3,
                            precision=stba.STBA_FP64)


def _run(ctx, s, room, iters, g):
    stba.stba_set_state(ctx, 0.3, 0.0, 0)
    stba.stba_set_params(ctx, s.cameras, s.points)
    stba.stba_record(ctx, room)
    for _ in range(iters):
        stba.stba_lm_iteration(ctx)
    out = [np.asarray(torch.as_tensor(x).cpu()) for x in stba.stba_adjoint(ctx, g)]
    if iters == room:
        with pytest.raises(stba.StbaError):
            stba.stba_lm_iteration(ctx)
    return out


@pytest.mark.parametrize("second", [(5, 3), (3, 3), (2, 2), (1, 1), (6, 2), (0, 0)])
def test_restarted_tape(second):
    m = 9
    clusters = (np.arange(m) * 3 // m).astype(np.int32)
    s = scenes.make_tiny_scene(m=m, n=60, seed=5, clusters=clusters, drop=0.3)
    g = np.random.default_rng(1).normal(size=(m, 9))
    room, iters = second
    with _ctx(s) as ctx, _ctx(s) as fresh:
        _run(ctx, s, 5, 2, g)
        if room == 0:
            stba.stba_record(ctx, 0)
            room = iters = 2
        got, want = _run(ctx, s, room, iters, g), _run(fresh, s, room, iters, g)
    for a, b in zip(got, want):
        assert np.max(np.abs(a - b)) <= 1e-8 * np.max(np.abs(b))
