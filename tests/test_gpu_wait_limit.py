"""The failure path of the device-side waits, without a fault: with a limit of 0 every wait of the factorisation and the
solves that does not find its data at the first look gives up.  The iteration comes back with failed clusters, is
rejected and leaves the parameters as they were; with the limit put back the next iteration is a fresh context's
(bars: the order of the atomic sums, 1e-9 in FP64; 1e-4 of each column in mixed precision, whose FP32 sums reach the
FP64 accumulators in a run-dependent order)."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

from elementwise import cols  # noqa: E402


def _scene(sizes=(35, 20, 40)):
    cl = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    return scenes.make_tiny_scene(m=len(cl), n=1000, seed=9, clusters=cl, drop=0.9)


def _ctx(s, **kw):
    return stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, s.clusters, lambda0=0.09, **kw)


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("precision,bar", [(stba.STBA_MIXED, 1e-4), (stba.STBA_FP64, 1e-9)])
def test_waits_that_run_out_reject_the_step(precision, bar, use_graph):
    s = _scene()
    with _ctx(s, precision=precision, use_graph=use_graph) as ctx, _ctx(s, precision=precision) as ref:
        for limit in (0, 0, 1_000_000_000):
            stba.stba_set_wait_limit(ctx, limit)
            stba.stba_set_state(ctx, 0.09, 0.0, 0)
            stba.stba_set_params(ctx, s.cameras, s.points)
            info = stba.stba_lm_iteration(ctx)
            if limit == 0:
                assert info["failed_clusters"] > 0 and not info["accepted"] and np.isinf(info["F_after"])
                c, p = stba.stba_get_params(ctx)
                assert np.array_equal(c, s.cameras) and np.array_equal(p, s.points)
        want = stba.stba_lm_iteration(ref)
        assert info["failed_clusters"] == 0 and info["accepted"] == want["accepted"]
        for a, b, w in zip(stba.stba_last_step(ctx), stba.stba_last_step(ref), (9, 3)):
            assert cols(a, b, w) < bar


@pytest.mark.parametrize("precision,bar", [(stba.STBA_MIXED, 1e-3), (stba.STBA_FP64, 1e-8)])
def test_waits_that_run_out_fail_the_adjoint(precision, bar):
    """STBA_ERR_TIMEOUT with the parameters as they were; the gradients of a fresh recording once the limit is back
    (bars of the adjoint's own tests: mixed 1e-3 of the largest entry; FP64 the order of the sums through two steps)."""
    s = _scene()
    g = np.random.default_rng(1).normal(size=(s.m, 9))
    with _ctx(s, precision=precision) as ctx, _ctx(s, precision=precision) as ref:
        for c in (ctx, ref):
            stba.stba_record(c, 2)
            for _ in range(2):
                assert stba.stba_lm_iteration(c)["accepted"]
        before = stba.stba_get_params(ctx)
        stba.stba_set_wait_limit(ctx, 0)
        with pytest.raises(stba.StbaError) as e:
            stba.stba_adjoint(ctx, g)
        assert e.value.status == 6
        after = stba.stba_get_params(ctx)
        assert np.array_equal(before[0], after[0]) and np.array_equal(before[1], after[1])
        stba.stba_set_wait_limit(ctx, 1_000_000_000)
        for a, b in zip(stba.stba_adjoint(ctx, g), stba.stba_adjoint(ref, g)):
            assert np.max(np.abs(a - b)) <= bar * np.max(np.abs(b))


def test_limits_out_of_range_are_refused():
    with _ctx(_scene((4, 4))) as ctx:
        for bad in (-1, 4_000_000_001):
            with pytest.raises(stba.StbaError):
                stba.stba_set_wait_limit(ctx, bad)
