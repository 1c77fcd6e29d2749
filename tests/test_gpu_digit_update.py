"""The update pass from digits on the tensor cores (tall merged cores) at the edges of its tiles (128 rows),
column groups (8, 16) and accumulators (FP64 32, FP32 48 and 64 outputs), on rows of very different sizes, and
over every kind of stencil column, against exact reconstruction and the oracle.  FP64 results agree to
1e-10 as every FP64 path does, the mixed path to 1e-5 (FP32 storage over three steps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt, problem  # noqa: E402
from paper_2602_00290_gb300.workloads import cube_config, plane_config1, random_tt, slab_config0  # noqa: E402

ROWS = 1024  # passes of at least this many rows may take the digits


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


@pytest.mark.parametrize("rows,rank", [(ROWS - 1, 9), (ROWS, 32), (ROWS + 1, 16), (ROWS + 127, 17), (ROWS + 129, 8),
                                       (ROWS + 64, 7), (ROWS + 3, 33), (ROWS + 5, 48), (ROWS + 31, 49), (ROWS, 64),
                                       (ROWS, 1), (152 * 128 * 2 + 9, 24)])
@pytest.mark.parametrize("prec,dtype,bar", [("fp64", "f64", 1e-10), ("mixed", "f64", 1e-5), ("mixed", "f32", 1e-5)])
def test_every_row_keeps_its_own_accuracy(tt, rows, rank, prec, dtype, bar):
    """Rows from 1 down to 2^-60: a rounding that drops nothing returns each to its own precision."""
    a = random_tt([rows, 70], [rank], seed=rows + rank)
    a[0] = a[0] * (2.0 ** -(61.0 * np.arange(rows) / rows).astype(int))[None, :, None]
    x = tt.TT.from_cores(a, rcap=[rank], dtype=dtype)
    ctx = tt.Context(0)
    tt.tt_round(ctx, x, 0.0, rank, prec)
    ctx.sync()
    got, want = nt.full(x.to_cores()), nt.full(a)
    err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() < bar


def test_scales_of_rows_and_columns_together(tt):
    a = random_tt([ROWS + 7, 70], [9], seed=5)
    cols, rows = 10.0 ** np.linspace(-100, 100, 9), 10.0 ** np.linspace(-90, 90, ROWS + 7)
    b = [a[0] * cols[None, None, :] * rows[None, :, None], a[1] / cols[:, None, None]]
    x = tt.TT.from_cores(b, rcap=[9])
    ctx = tt.Context(0)
    tt.tt_round(ctx, x, 0.0, 9)
    ctx.sync()
    got, want = nt.full(x.to_cores()) / rows[:, None], nt.full(a)
    live = rows > 1e90 * 1e-12  # columns of the factor are resolved to about 2^-57 of their largest entry
    assert np.max(np.abs(got - want)[live]) < 1e-10 * np.max(np.abs(want))
    assert np.all(np.isfinite(got))


@pytest.mark.parametrize("prec,dtype", [("fp64", "f64"), ("mixed", "f32")])
def test_nonfinite_rows_are_reported(tt, prec, dtype):
    a = random_tt([ROWS, 70], [8], seed=1)
    a[0][0, ROWS - 3, 5] = np.nan
    x = tt.TT.from_cores(a, rcap=[8], dtype=dtype)
    ctx = tt.Context(0)
    tt.tt_round(ctx, x, 0.0, 8, prec)
    with pytest.raises(tt.TTError) as e:
        ctx.sync()
    assert e.value.status == tt.TT_ERR_NONFINITE


FACES = (0.9, 0.4, 0.6, 0.8, None, None)
PLANE = dict(nx=38, ny=37, G=12, ntheta=4, nphi=8, tol=1e-8)
CASES = [
    dict(wl=lambda: plane_config1(rmax=12, **PLANE)),
    dict(wl=lambda: plane_config1(rmax=9, **PLANE).with_(inflow_temperature=FACES)),
    dict(wl=lambda: plane_config1(rmax=12, **PLANE).with_(flux="rusanov")),
    dict(wl=lambda: plane_config1(rmax=8, **PLANE).with_(flux="central")),
    dict(wl=lambda: cube_config(nx=14, ny=13, nz=12, G=8, rmax=10, tol=1e-8).with_(
        inflow_temperature=(0.9, None, None, 0.5, 0.7, None))),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("prec,dtype,bar", [("fp64", "f64", 1e-10), ("mixed", "f32", 1e-5), ("mixed", "f64", 1e-5)])
def test_step_matches_the_oracle(tt, case, prec, dtype, bar):
    wl = CASES[case]["wl"]()
    coef = problem.build(wl)
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, wl)
    x = tt.initial_state(plan, [wl.rmax] * (plan.d - 1), dtype)
    assert x.n[0] > 128 * 128
    ref = nt.initial_tt(problem.initial_rows(wl, coef), coef)
    for _ in range(3):
        tt.tt_step(ctx, plan, x, wl.tol, wl.rmax, prec)
        ref = nt.step(ref, coef, wl.tol, wl.rmax)
    E = tt.tt_energy_density(ctx, plan, x)
    ctx.sync()
    want = nt.energy_density_rows(ref, coef)
    assert np.linalg.norm(E.cpu().numpy().ravel() - want.ravel()) <= bar * np.linalg.norm(want)
    if prec == "fp64":
        assert x.ranks() == nt.ranks(ref)
        got, full = nt.to_dense_rows(x.to_cores()), nt.to_dense_rows(ref)
        assert np.max(np.abs(got - full)) <= bar * np.max(np.abs(full))
