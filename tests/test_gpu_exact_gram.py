"""The triangular factor from exact Gram products (the default factor of every rounding) at the edges
of its column groups (8, 16, 32 columns), row octets and tiles (8, 64 rows) and cells (groups per cell
not a multiple of 8), against the Householder kernels (chosen with tt_context_set_tsqr) and exact
reconstruction.  FP64 results agree to 1e-10 as every FP64 path does; the mixed path to 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt  # noqa: E402
from paper_2602_00290_gb300.workloads import cube_config, plane_config1, random_tt, slab_config0  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def rel(a, b):
    return float(np.max(np.abs(a - b))) / max(float(np.max(np.abs(b))), 1e-300)


def householder(ctx):
    for prec in ("fp64", "mixed"):
        for n in range(1, 257):
            ctx.set_tsqr(prec, n, "column", 0)


@pytest.mark.parametrize("rows", [1, 7, 9, 64, 65, 1037])
@pytest.mark.parametrize("rank", [1, 8, 9, 16, 17, 32, 33, 40])
def test_exact_rank_round_reconstructs(tt, rows, rank):
    a = random_tt([rows, 6, 7], [rank, 7], seed=100 * rows + rank)
    ctx = tt.Context(0)
    for prec, dtype, bar in (("fp64", "f64", 1e-10), ("mixed", "f64", 1e-5), ("mixed", "f32", 1e-5)):
        x = tt.TT.from_cores(a, rcap=[rank, 7], dtype=dtype)
        tt.tt_round(ctx, x, 0.0, min(rank, 7), prec)
        ctx.sync()
        y = tt.TT.from_cores(a, rcap=[rank, 7], dtype=dtype)
        other = tt.Context(0)
        householder(other)
        tt.tt_round(other, y, 0.0, min(rank, 7), prec)
        other.sync()
        assert x.ranks() == y.ranks()
        assert rel(nt.full(x.to_cores()), nt.full(y.to_cores())) < bar, (prec, dtype)


def test_columns_of_very_different_scales(tt):
    """Columns 1e-120 .. 1e120 apart, with the right part scaled back: each has its own fixed point."""
    a = random_tt([300, 6, 7], [9, 7], seed=3)
    scale = 10.0 ** np.linspace(-120, 120, 9)
    b = [a[0] * scale[None, None, :], a[1] / scale[:, None, None], a[2]]
    ctx = tt.Context(0)
    x = tt.TT.from_cores(b, rcap=[9, 7])
    tt.tt_round(ctx, x, 1e-13, 7)
    ctx.sync()
    want = nt.full(nt.round_tt(a, 1e-13, 7))
    assert rel(nt.full(x.to_cores()), want) < 1e-10


CASES = [
    dict(wl=lambda G: slab_config0().with_(rmax=6, tol=1e-8), G=16),
    dict(wl=lambda G: plane_config1(nx=7, ny=5, G=G, ntheta=4, nphi=8, rmax=8, tol=1e-8), G=1),
    dict(wl=lambda G: plane_config1(nx=9, ny=6, G=G, ntheta=4, nphi=8, rmax=8, tol=1e-8).with_(
        inflow_temperature=(0.9, 0.4, 0.6, 0.8, None, None)), G=7),
    dict(wl=lambda G: plane_config1(nx=6, ny=7, G=G, ntheta=4, nphi=8, rmax=5, tol=1e-8).with_(flux="rusanov"), G=8),
    dict(wl=lambda G: plane_config1(nx=6, ny=7, G=G, ntheta=4, nphi=8, rmax=8, tol=1e-8).with_(flux="central"), G=9),
    dict(wl=lambda G: cube_config(nx=4, ny=5, nz=3, G=G, rmax=8, tol=1e-8).with_(
        inflow_temperature=(0.9, None, None, 0.5, 0.7, None)), G=3),
    dict(wl=lambda G: cube_config(nx=5, ny=1, nz=4, G=G, rmax=8, tol=1e-8), G=17),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("prec,dtype,bar", [("fp64", "f64", 1e-10), ("mixed", "f32", 2e-6), ("mixed", "f64", 2e-6)])
def test_step_agrees_with_the_householder_factor(tt, case, prec, dtype, bar):
    wl = CASES[case]["wl"](CASES[case]["G"])
    out = []
    for kernels in ("exact", "householder"):
        ctx = tt.Context(0)
        if kernels == "householder":
            householder(ctx)
        plan = tt.Plan(ctx, wl)
        x = tt.initial_state(plan, [wl.rmax] * (plan.d - 1), dtype)
        for _ in range(3):
            tt.tt_step(ctx, plan, x, wl.tol, wl.rmax, prec)
        E = tt.tt_energy_density(ctx, plan, x)
        ctx.sync()
        out.append((x.ranks(), E.cpu().numpy(), nt.to_dense_rows(x.to_cores())))
    (r0, e0, f0), (r1, e1, f1) = out
    assert np.linalg.norm(e0 - e1) <= bar * np.linalg.norm(e1)
    if prec == "fp64":
        assert r0 == r1
        assert rel(f0, f1) < bar


def test_step_captured_on_a_workspace_of_the_householder_size(tt):
    """A capture cannot grow the workspace: one that only holds the Householder factors still steps."""
    wl = plane_config1(nx=24, ny=20, G=6, ntheta=4, nphi=8, rmax=8, tol=1e-6)
    small = tt.Context(0)
    householder(small)
    plan = tt.Plan(small, wl)
    x = tt.initial_state(plan, [8, 8], "f64")
    tt.tt_step(small, plan, x, wl.tol, wl.rmax, "fp64")
    small.sync()
    need = tt.tt_workspace_query(small, plan, x, "fp64")
    stream = torch.cuda.Stream()
    ctx = tt.Context(0, stream=stream, workspace_bytes=need)
    assert tt.tt_workspace_query(ctx, plan, x, "fp64") > need
    y = tt.initial_state(plan, [8, 8], "f64")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        tt.tt_step(ctx, plan, y, wl.tol, wl.rmax, "fp64")
    graph.replay()
    torch.cuda.synchronize()
    ctx.sync()
    assert y.ranks() == x.ranks()
    assert rel(nt.to_dense_rows(y.to_cores()), nt.to_dense_rows(x.to_cores())) < 1e-10
