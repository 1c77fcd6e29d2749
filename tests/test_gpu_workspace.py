"""The context's workspace over calls of different need: a graph that the caller captured keeps the workspace it
was captured on, whatever larger one later calls take, and a workspace that the device refuses is asked for once.
Steps agree with steps on an ample workspace to 1e-10 (FP64)."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt  # noqa: E402
from paper_2602_00290_gb300.workloads import plane_config1, random_tt  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WL = plane_config1(nx=24, ny=20, G=6, ntheta=4, nphi=8, rmax=8, tol=1e-6)


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def dense(x):
    return nt.to_dense_rows(x.to_cores())


def reference(tt, steps):
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, WL)
    x = tt.initial_state(plan, [8, 8], "f64")
    for _ in range(steps):
        tt.tt_step(ctx, plan, x, WL.tol, WL.rmax)
    ctx.sync()
    return dense(x)


def close(got, want):
    return np.max(np.abs(got - want)) < 1e-10 * np.max(np.abs(want))


def small_need(tt):
    ctx = tt.Context(0)
    for n in range(1, 257):
        ctx.set_tsqr("fp64", n, "column", 0)
    plan = tt.Plan(ctx, WL)
    x = tt.initial_state(plan, [8, 8], "f64")
    tt.tt_step(ctx, plan, x, WL.tol, WL.rmax)
    ctx.sync()
    return tt.tt_workspace_query(ctx, plan, x)


@pytest.mark.parametrize("grow", ["dot", "step"])
def test_captured_step_survives_a_larger_workspace(tt, grow):
    stream = torch.cuda.Stream()
    ctx = tt.Context(0, stream=stream, workspace_bytes=small_need(tt) if grow == "step" else 0)
    plan = tt.Plan(ctx, WL)
    x = tt.initial_state(plan, [8, 8], "f64")
    if grow == "dot":  # every kernel is loaded, and the workspace sized, before the capture
        y = tt.initial_state(plan, [8, 8], "f64")
        tt.tt_step(ctx, plan, y, WL.tol, WL.rmax)
        ctx.sync()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        tt.tt_step(ctx, plan, x, WL.tol, WL.rmax)
    graph.replay()
    torch.cuda.synchronize()
    ctx.sync()
    assert close(dense(x), reference(tt, 1))
    # a call that needs more, and what takes the memory that a freed workspace would leave
    if grow == "dot":
        a = tt.TT.from_cores(random_tt([200000, 6], [32], seed=1))
        tt.tt_dot(ctx, a, a)
    else:
        z = tt.initial_state(plan, [8, 8], "f64")
        tt.tt_step(ctx, plan, z, WL.tol, WL.rmax)
    ctx.sync()
    assert tt.tt_workspace_query(ctx, plan, x) > 0
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    ctx.sync()
    assert close(dense(x), reference(tt, 3))
    ctx.close()


SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <stdlib.h>
static long calls;
long tt_shim_calls(void) { return calls; }
int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t);
  if (!real) real = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
  const char* most = getenv("TT_SHIM_MOST");
  ++calls;
  if (most && n > (size_t)atol(most)) return 2; /* cudaErrorMemoryAllocation */
  return real(p, n);
}
"""
SCRIPT = """
import ctypes, os
import numpy as np
import torch
import paper_2602_00290_gb300 as tt
from paper_2602_00290_gb300.workloads import plane_config1
wl = plane_config1(nx=128, ny=128, G=16, ntheta=4, nphi=8, rmax=8, tol=1e-6)
calls = ctypes.CDLL(None).tt_shim_calls
calls.restype = ctypes.c_long
def steps(most, graphs):
    os.environ.pop("TT_SHIM_MOST", None)
    ctx = tt.Context(0)
    ctx.set_graphs(graphs)
    plan = tt.Plan(ctx, wl)
    x = tt.initial_state(plan, [8, 8], "f64")
    out = tt.tt_energy_density(ctx, plan, x)
    torch.cuda.synchronize()
    if most:
        assert tt.tt_workspace_query(ctx, plan, x) > most
        ctypes.CDLL(None).setenv(b"TT_SHIM_MOST", str(most).encode(), 1)
    n = []
    for _ in range(10):
        before = calls()
        tt.tt_step(ctx, plan, x, wl.tol, wl.rmax)
        n.append(calls() - before)
    ctypes.CDLL(None).unsetenv(b"TT_SHIM_MOST")
    tt.tt_energy_density(ctx, plan, x, out)
    ctx.sync()
    return n, out.cpu().numpy()
free, want = steps(0, False)
assert sum(free[1:]) == 0 and free[0] > 0, free
for graphs in (False, True):
    n, got = steps(100 << 20, graphs)
    assert 1 < n[0] <= 4 and sum(n[1:]) == 0, n
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
"""


def test_a_refused_workspace_is_asked_for_once(tt, tmp_path):
    gcc = shutil.which("gcc")
    if not gcc:
        pytest.skip("needs gcc")
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run([gcc, "-shared", "-fPIC", "-O1", str(src), "-o", str(lib), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=str(lib)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
