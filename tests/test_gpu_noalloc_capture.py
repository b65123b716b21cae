"""stba_cost_noalloc inside a captured graph (its launches carry programmatic dependencies): replays give the eager
call's value bit for bit, for the captured inputs and after they have changed."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


def test_noalloc_cost_in_a_captured_graph():
    s = scenes.make_tiny_scene(m=20, n=500, seed=1, drop=0.3)
    t = [torch.as_tensor(x).cuda() for x in (s.cameras, s.points, s.obs_cam.astype(np.int32), s.obs_pt.astype(np.int32),
                                             s.obs_uv)]
    F = torch.zeros(1, dtype=torch.float64, device="cuda")
    stba.stba_cost_noalloc(*t, F)   # the first call, before any capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(2):
            stba.stba_cost_noalloc(*t, F)
    for shift in (0.0, 0.01, 0.01):
        t[0][:, 3] += shift
        stba.stba_cost_noalloc(*t, F)
        want = F.item()
        F.zero_()
        graph.replay()
        assert F.item() == want
