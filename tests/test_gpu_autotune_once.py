"""stba_autotune times a configuration once: the tensor-core steps have one panel, so the split and the stacked name of
it share a time and the stacked one is the one kept."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402


def test_one_configuration_is_timed_once():
    cl = (np.arange(40) // 20).astype(np.int32)
    s = scenes.make_tiny_scene(m=40, n=300, seed=4, clusters=cl, drop=0.8)
    with stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, cl, precision=stba.STBA_MIXED) as ctx:
        kept, ms = stba.stba_autotune(ctx, 4)
        assert ms["64_split_tensor"] == ms["64_stacked_tensor"] > 0
        assert kept != "64_split_tensor" and ms[kept] == min(ms.values())
