"""The start and the end of an iteration (tables, zeros, step scatter, stop-test sums, candidate cost, accept) at
the edges of their grids: 32 cameras per table block, 256 points per CTA, and 256 observations per SM, up to which
the launches of an iteration are chained.  Two iterations, each checked against FP64 formulas on the step that the
device returns.  Tolerances: the norms are FP64 sums of at most 4000 squares (1e-11); the FP64 cost 1e-10 (the mixed
cost rounds its distortion term to FP32; the parity tests cover it); the gradient is a sum of FP32 (FP64) products,
each within 1e-5 (1e-12) of itself; an accepted step is added in FP64, exactly; the residuals of the accepted
candidate, stored for the next linearisation, show in the next iteration's gradient."""
import numpy as np
import pytest

import scenes
from oracle import camera as ocam
from oracle import stba as ostba

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


def _chain_limit():
    return 256 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("size", [(3, 11), (31, 255), (32, 256), (33, 257), "below", "above"])
def test_iteration_start_and_end(size, precision, graph):
    m, n = size if isinstance(size, tuple) else (32, _chain_limit() // 32 + (size == "above"))
    cl = (np.arange(m) * 3 // m).astype(np.int32)
    s = scenes.make_tiny_scene(m=m, n=n, seed=m, clusters=cl, drop=0.0)
    obs = (s.obs_cam, s.obs_pt, s.obs_uv)
    mixed = precision == "mixed"
    with stba.stba_create(s.cameras, s.points, *obs, cl, lambda0=0.09, use_graph=graph,
                          precision=stba.STBA_MIXED if mixed else stba.STBA_FP64) as ctx:
        for it in range(2):
            c0, p0 = stba.stba_get_params(ctx)
            c0, p0 = np.array(c0).reshape(m, 9), np.array(p0).reshape(n, 3)
            lam = stba.stba_get_state(ctx)[0]
            info = stba.stba_lm_iteration(ctx)
            dc, dp = stba.stba_last_step(ctx)
            dc, dp = np.asarray(dc).reshape(m, 9), np.asarray(dp).reshape(n, 3)
            c1, p1 = stba.stba_get_params(ctx)
            assert info["lambda_used"] == lam and info["iteration"] == it + 1 and info["failed_clusters"] == 0
            assert abs(info["dx_norm"] / np.sqrt(np.sum(dc**2) + np.sum(dp**2)) - 1) < 1e-11
            assert abs(info["x_norm"] / np.sqrt(np.sum(c0**2) + np.sum(p0**2)) - 1) < 1e-11
            F = [ocam.cost(c0, p0, *obs), ocam.cost(c0 + dc, p0 + dp, *obs)]
            if not mixed:
                for got, want in zip((info["F_before"], info["F_after"]), F):
                    assert abs(got / want - 1) < 1e-10
            assert info["accepted"] == (F[1] < F[0])
            step = (c0 + dc, p0 + dp) if info["accepted"] else (c0, p0)
            assert np.array_equal(np.asarray(c1).reshape(m, 9), step[0])
            assert np.array_equal(np.asarray(p1).reshape(n, 3), step[1])
            f = ocam.residuals(c0, p0, *obs)
            Jc, Jp = ocam.jacobians(c0, p0, s.obs_cam, s.obs_pt)
            g, size_g = [], []
            for J, ids, k in ((Jc, s.obs_cam, m), (Jp, s.obs_pt, n)):
                t = np.einsum("oij,oi->oj", J, f)
                a = np.einsum("oij,oi->oj", np.abs(J), np.abs(f))
                for acc, val in ((g, t), (size_g, a)):
                    out = np.zeros((k, J.shape[2]))
                    np.add.at(out, ids, val)
                    acc.append(out.ravel())
            g, size_g = np.abs(np.concatenate(g)), np.concatenate(size_g)
            i = np.argmax(g)
            assert abs(info["grad_inf"] - g[i]) <= (1e-5 if mixed else 1e-12) * max(size_g[i], size_g[np.argmax(size_g)])
