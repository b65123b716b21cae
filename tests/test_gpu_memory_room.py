"""Buffers that a context holds for speed alone give way when another allocation finds no room: FP64 rows stored by
default, the PCG Jacobians in slot order, the split operands of the tensor-core steps.  The room is limited on the
host, in a child process whose cudaMalloc and cudaMemGetInfo go through a preloaded counter; nothing is filled.  The
step is that of a context with room (order of the FP64 atomic sums: 1e-9 of each column; CG stopped at 1e-12: 1e-7;
mixed precision 1e-4)."""
import os
import subprocess
import sys
import textwrap

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#define N 65536
static void* ptr[N]; static size_t len[N]; static size_t used, limit = (size_t)-1; static int n;
void room(size_t more) { limit = used + more; }   /* bytes that may still be allocated */
void no_limit(void) { limit = (size_t)-1; }
int cudaMalloc(void** p, size_t bytes) {
  static int (*real)(void**, size_t);
  if (!real) real = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
  if (limit != (size_t)-1 && used + bytes > limit) return 2;   /* cudaErrorMemoryAllocation */
  int e = real(p, bytes);
  if (!e && n < N) { ptr[n] = *p; len[n++] = bytes; used += bytes; }
  return e;
}
int cudaFree(void* p) {
  static int (*real)(void*);
  if (!real) real = (int (*)(void*))dlsym(RTLD_NEXT, "cudaFree");
  for (int i = 0; p && i < n; ++i) if (ptr[i] == p) { used -= len[i]; ptr[i] = ptr[--n]; len[i] = len[n]; break; }
  return real(p);
}
int cudaMemGetInfo(size_t* f, size_t* t) {
  static int (*real)(size_t*, size_t*);
  if (!real) real = (int (*)(size_t*, size_t*))dlsym(RTLD_NEXT, "cudaMemGetInfo");
  int e = real(f, t);
  if (!e && limit != (size_t)-1) { *f = limit - used; }
  return e;
}
"""

CHILD = """
    import ctypes, sys
    sys.path[:0] = [{root!r}, {tests!r}]
    import numpy as np
    import scenes
    from elementwise import cols
    from paper_2008_00446_gb300 import stba
    shim = ctypes.CDLL({shim!r})
    shim.room.argtypes = [ctypes.c_size_t]
    s = scenes.make_tiny_scene(m=300, n=1000, seed=2, drop=0.9)
    one, many = np.zeros(300, np.int32), (np.arange(300) // 10).astype(np.int32)
    def make(cl=one, **kw):
        kw.setdefault("precision", stba.STBA_FP64)
        return stba.stba_create(s.cameras, s.points, s.obs_cam, s.obs_pt, s.obs_uv, cl, lambda0=0.09, **kw)
    def size(ctx):
        return stba.stba_problem_info(ctx)["device_bytes"]
    def step(ctx):
        stba.stba_lm_iteration(ctx)
        return stba.stba_last_step(ctx)
    def same(a, b, bar):
        for x, y, w in zip(a, b, (9, 3)):
            assert cols(x, y, w) < bar, cols(x, y, w)
    with make() as c:   # one-time allocations of the process and the modules
        step(c)
"""

ROWS = """
    rows = 24 * 8 * len(s.obs_cam)
    with make(pair_blocks=stba.STBA_PAIR_BLOCKS_RECOMPUTE) as ref, make() as roomy:
        need, want = size(ref), step(ref)
        assert size(roomy) > need + rows // 2     # the default stores the rows
    shim.room(need + rows // 2)
    with make() as ctx:
        assert size(ctx) < need + rows // 2
        same(step(ctx), want, 1e-9)
    with make(many) as ctx:                       # stored at create, given up for a larger assignment
        small = size(ctx)
        step(ctx)
        stba.stba_set_params(ctx, s.cameras, s.points)
        stba.stba_set_state(ctx, 0.09)
        stba.stba_set_clusters(ctx, one)
        same(step(ctx), want, 1e-9)
    shim.room(need + rows // 2)
    try:
        make(pair_blocks=stba.STBA_PAIR_BLOCKS_STORED)
        raise SystemExit("stored rows fitted")
    except stba.StbaError as e:
        assert e.status == 3
"""

PCG = """
    for solver in (stba.STBA_SOLVER_PCG_FULL, stba.STBA_SOLVER_PCG_CLUSTERS):
        for precision, real, bar in ((stba.STBA_FP64, 8, 1e-7), (stba.STBA_MIXED, 4, 1e-4)):
            kw = dict(linear_solver=solver, precision=precision, pcg_tol=1e-12 if real == 8 else 1e-7, pcg_max_iter=200)
            shim.no_limit()
            with make(many, **kw) as ref:
                need, want = size(ref), step(ref)
            copy = 24 * real * len(s.obs_cam)
            shim.room(need - copy // 2)
            with make(many, **kw) as ctx:
                assert size(ctx) < need - copy // 2
                same(step(ctx), want, bar)
"""

SPLIT = """
    with make(precision=stba.STBA_MIXED, factor_update=stba.STBA_FACTOR_UPDATE_SIMT) as ref:
        need, want = size(ref), step(ref)
    with make(precision=stba.STBA_MIXED) as roomy:
        assert size(roomy) > need + 2 * 1024 * 1024
    shim.room(need + 1024 * 1024)
    with make(precision=stba.STBA_MIXED) as ctx:
        same(step(ctx), want, 1e-4)
"""


@pytest.mark.parametrize("body", [ROWS, PCG, SPLIT], ids=["fp64_rows", "pcg_slots", "split_operands"])
def test_without_room_for_optional_buffers(tmp_path, body):
    tests = os.path.dirname(os.path.abspath(__file__))
    src, shim, script = tmp_path / "room.c", tmp_path / "libroom.so", tmp_path / "child.py"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", str(src), "-o", str(shim), "-ldl"], check=True)
    script.write_text(textwrap.dedent(CHILD).format(root=os.path.dirname(tests), tests=tests, shim=str(shim)) +
                      textwrap.dedent(body))
    r = subprocess.run([sys.executable, str(script)], env=dict(os.environ, LD_PRELOAD=str(shim)), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
