"""The digit update (tall merged cores) under the rounding methods whose factor does not carry every column at
its own size: Gram rounding, whose factor ends at pivots of 4 n eps of the largest diagonal entry, and
randomized rounding, whose factor holds the columns' parts inside the sketch.  States of mutually orthogonal
columns graded over twelve decades or more.

Bars, in units of the state's Frobenius norm.  Gram: the columns that the factor leaves out are below
sqrt(4 n eps) <= 2e-7 for n <= 45 columns, together below 2e-7 sqrt(9): 1e-6, and 1e-5 with FP32 storage.
Randomized, against the oracle with the same sketch: 1e-10 as every FP64 path, 1e-5 mixed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt, problem  # noqa: E402
from paper_2602_00290_gb300.workloads import plane_config1, sketch_matrix  # noqa: E402

ROWS = 1531
PRECS = [("fp64", "f64"), ("mixed", "f32"), ("mixed", "f64")]


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def graded(rows, modes, grades, seed):
    """Orthonormal columns times `grades`, orthonormal right parts."""
    rng = np.random.default_rng(seed)
    r = len(grades)
    q = np.linalg.qr(rng.standard_normal((rows, r)))[0] * np.asarray(grades)[None, :]
    cores = [q[None]]
    for j, n in enumerate(modes):
        r1 = r if j < len(modes) - 1 else 1
        w = np.linalg.qr(rng.standard_normal((n * r1, r)))[0].T
        cores.append(w.reshape(r, n, r1))
    return cores


def err(got, want):
    return np.linalg.norm(got - want) / np.linalg.norm(want)


@pytest.mark.parametrize("prec,dtype", PRECS)
def test_gram_round_of_graded_columns(tt, prec, dtype):
    a = graded(ROWS, [70], np.logspace(0, -12, 9), seed=1)
    ctx = tt.Context(0)
    ctx.set_rounding("gram")
    x = tt.TT.from_cores(a, rcap=[9], dtype=dtype)
    tt.tt_round(ctx, x, 0.0, 9, prec)
    ctx.sync()
    assert err(nt.full(x.to_cores()), nt.full(a)) < (1e-6 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("prec,dtype", PRECS)
@pytest.mark.parametrize("faces", [None, (0.9, None, 0.6, None, None, 0.7)])
def test_gram_step_of_graded_columns(tt, prec, dtype, faces):
    wl = plane_config1(nx=14, ny=11, G=9, ntheta=4, nphi=10, rmax=9, tol=1e-5)
    if faces:
        wl = wl.with_(inflow_temperature=faces)
    coef = problem.build(wl)
    a = graded(wl.nrow, [4, 10], np.logspace(0, -12, 9), seed=2)
    ctx = tt.Context(0)
    ctx.set_rounding("gram")
    plan = tt.Plan(ctx, wl)
    x = tt.TT.from_cores(a, rcap=[9, 9], dtype=dtype)
    tt.tt_step(ctx, plan, x, wl.tol, wl.rmax, prec)
    ctx.sync()
    ref = nt.step(a, coef, wl.tol, wl.rmax, rounding="gram")
    assert err(nt.full(x.to_cores()), nt.full(ref)) < (1e-6 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("prec,dtype", PRECS)
def test_randomized_round_of_graded_columns(tt, prec, dtype):
    # eight columns that a sketch of eight holds and four far outside it
    grades = list(0.5 ** np.arange(8)) + [1e-9, 1e-12, 1e-15, 1e-18]
    a = graded(ROWS, [70], grades, seed=3)
    om = sketch_matrix(70, 8, seed=5)
    ctx = tt.Context(0)
    ctx.set_sketch(om)
    ctx.set_rounding("randomized")
    x = tt.TT.from_cores(a, rcap=[12], dtype=dtype)
    tt.tt_round(ctx, x, 1e-6, 12, prec)
    ctx.sync()
    want = nt.round_tt_randomized(a, 1e-6, 12, om)
    assert x.ranks() == nt.ranks(want)
    assert err(nt.full(x.to_cores()), nt.full(want)) < (1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("prec,dtype", PRECS)
def test_randomized_step_of_graded_columns(tt, prec, dtype):
    wl = plane_config1(nx=14, ny=11, G=9, ntheta=4, nphi=10, rmax=9, tol=1e-5)
    coef = problem.build(wl)
    a = graded(wl.nrow, [4, 10], np.logspace(0, -12, 9), seed=4)
    om = sketch_matrix(40, 16, seed=7)
    ctx = tt.Context(0)
    ctx.set_sketch(om)
    ctx.set_rounding("randomized")
    plan = tt.Plan(ctx, wl)
    x = tt.TT.from_cores(a, rcap=[9, 9], dtype=dtype)
    tt.tt_step(ctx, plan, x, wl.tol, wl.rmax, prec)
    ctx.sync()
    ref = nt.step(a, coef, wl.tol, wl.rmax, rounding="randomized", omega=om)
    assert err(nt.full(x.to_cores()), nt.full(ref)) < (1e-10 if prec == "fp64" else 1e-5)
