"""Rounding errors of the FP32 cluster factor and solve, without refinement: the step's distance from an FP64 solve of
the device's own S' and b', over four systems of 1080 unknowns at lambda = 0.05, against that of a factor made on the
host with the same rounding (fused multiply-adds, tiles of 64, columns in blocks of 8, every sum of products from zero)
and solved in FP64.  The device's two triangular passes add about as much independent rounding again: 1.41 times the
host's error.  Where the products come off an entry one by one, which rounds eight times as often at the entry's
magnitude, the host's own factor is 1.86 times worse, so the step 2.11 times.  Bar: 1.73, their geometric mean."""
import numpy as np
import pytest
import scipy.linalg as sl

import scenes
from oracle import camera as ocam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2008_00446_gb300 import stba  # noqa: E402

M = 120


def _scene(seed):
    """points around the origin, each seen by 6 cameras of a window of 16"""
    rng = np.random.default_rng(seed)
    base = scenes.make_tiny_scene(m=M, n=64, seed=3, drop=0.9)
    n = 8 * M
    oc = (np.arange(n)[:, None] * M // n + rng.permuted(np.tile(np.arange(16), (n, 1)), axis=1)[:, :6]) % M
    oc = np.sort(oc, 1).ravel().astype(np.int32)
    op = np.repeat(np.arange(n), 6).astype(np.int32)
    pts = rng.uniform(-0.3, 0.3, (n, 3))
    uv = ocam.residuals(base.cameras_true, pts, oc, op, np.zeros((len(oc), 2))) + rng.normal(0, 1, (len(oc), 2))
    return base.cameras, pts, oc, op, uv


def _fma(a, b, c):   # a product of two FP32 values is exact in FP64
    return (a.astype(np.float64) * b + c).astype(np.float32)


def _factor(A):
    """LL^T of A in FP32"""
    n, A = len(A), A.astype(np.float32)
    for k0 in range(0, n, 64):
        k1 = min(k0 + 64, n)
        for c in range(k0, k1):
            b0 = k0 + (c - k0) // 8 * 8
            v = A[c:, c].copy()
            for t0 in range(k0, b0, 8):
                s = np.zeros_like(v)
                for t in range(t0, t0 + 8):
                    s = _fma(A[c:, t], A[c, t], s)
                v = v - s
            for t in range(b0, c):
                v = _fma(-A[c:, t], A[c, t], v)
            A[c:, c] = v * (np.float32(1) / np.sqrt(v[0]))
        s = np.zeros_like(A[k1:, k1:])
        for t in range(k0, k1):
            s = _fma(A[k1:, t, None], A[None, k1:, t], s)
        A[k1:, k1:] -= s
    return np.tril(A).astype(np.float64)


@pytest.mark.parametrize("update", [stba.STBA_FACTOR_UPDATE_TENSOR, stba.STBA_FACTOR_UPDATE_SIMT])
def test_unrefined_step_rounds_as_fp32_sums_do(update):
    here, host = [], []
    for seed in range(4):
        with stba.stba_create(*_scene(seed), np.zeros(M, np.int32), lambda0=0.05, precision=stba.STBA_MIXED,
                              refine_steps=0, factor_update=update) as ctx:
            stba.stba_lm_iteration(ctx)
            dc, _ = stba.stba_last_step(ctx)
            S, b = stba.stba_get_cluster_system(ctx, 0)
        d = 1 / np.sqrt(np.diag(S))
        A, r = S * d[:, None] * d, b * d
        z = sl.cho_solve(sl.cho_factor(A, lower=True), r)
        here.append(np.linalg.norm(dc.ravel() / d - z) / np.linalg.norm(z))
        host.append(np.linalg.norm(sl.cho_solve((_factor(A), True), r) - z) / np.linalg.norm(z))
    assert np.mean(here) < 1.73 * np.mean(host), (here, host)
