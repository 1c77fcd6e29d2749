"""Inner products and the materialised transport sum on tall cores: the inner product's exact products (from
16,384 rows; passes of 262,144 rows; groups of 16 columns) against FP64 sums to 1e-12 of the norms, and
the FP32 transport sum against its FP64 form, rounded: one unit in the last place, at every size of entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt  # noqa: E402
from paper_2602_00290_gb300.workloads import cube_config, plane_config1, random_tt  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


@pytest.mark.parametrize("rows,rx,ry", [(16383, 5, 7), (16384, 32, 32), (16385, 17, 5), (16384 + 63, 33, 8),
                                        (20000, 1, 1), ((1 << 18) + 77, 3, 4)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_dot_of_tall_cores(tt, rows, rx, ry, dtype):
    a, b = random_tt([rows, 40], [rx], seed=rows), random_tt([rows, 40], [ry], seed=rows + 1)
    if dtype == "f32":
        a, b = ([c.astype(np.float32).astype(np.float64) for c in t] for t in (a, b))
    x, y = tt.TT.from_cores(a, rcap=[rx + 1], dtype=dtype), tt.TT.from_cores(b, rcap=[ry], dtype=dtype)
    ctx = tt.Context(0)
    for u, v, p, q in ((x, y, a, b), (x, x, a, a), (y, x, b, a)):
        want = float(np.sum(nt.full(p) * nt.full(q)))
        assert abs(tt.tt_dot(ctx, u, v).item() - want) <= 1e-12 * nt.norm(p) * nt.norm(q)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_dot_keeps_what_is_not_finite(tt, value):
    a, b = random_tt([16400, 40], [6], seed=1), random_tt([16400, 40], [6], seed=2)
    a[0][0, 16399, 2] = value
    x, y = tt.TT.from_cores(a, rcap=[6]), tt.TT.from_cores(b, rcap=[6])
    assert not np.isfinite(tt.tt_dot(tt.Context(0), x, y).item())
    assert np.isfinite(tt.tt_dot(tt.Context(0), y, y).item())


@pytest.mark.parametrize("dtype,scale", [("f64", 1.0), ("f64", 1e-280), ("f32", 1.0), ("f32", 1e-30)])
def test_dot_of_fields_that_are_large_on_different_rows(tt, dtype, scale):
    # positive entries: an FP64 sum is within (rows + angles) 2^-53 = 1.9e-12 of the value, twice that for both sides
    rng = np.random.default_rng(5)
    rows, far = 16400, np.arange(16400) < 8200
    a = [scale * rng.uniform(0.5, 1.0, (1, rows, 3)) * np.where(far, 1.0, 1e-12)[None, :, None], rng.uniform(0.5, 1.0, (3, 40, 1))]
    b = [rng.uniform(0.5, 1.0, (1, rows, 2)) * np.where(far, 1e-12, 1.0)[None, :, None], rng.uniform(0.5, 1.0, (2, 40, 1))]
    if dtype == "f32":
        a, b = ([c.astype(np.float32).astype(np.float64) for c in t] for t in (a, b))
    x, y = tt.TT.from_cores(a, rcap=[3], dtype=dtype), tt.TT.from_cores(b, rcap=[2], dtype=dtype)
    want = float(np.sum((a[0][0].T @ b[0][0]) * (a[1][:, :, 0] @ b[1][:, :, 0].T)))
    assert abs(tt.tt_dot(tt.Context(0), x, y).item() - want) <= 4e-12 * want


WORKLOADS = [
    (plane_config1(nx=9, ny=7, G=5, ntheta=4, nphi=8, rmax=8).with_(
        inflow_temperature=(0.9, None, 0.6, None, None, 0.7)), 8, 48),
    (plane_config1(nx=9, ny=7, G=16, ntheta=4, nphi=8, rmax=60), 60, 300),
    (plane_config1(nx=17, ny=4, G=3, ntheta=4, nphi=8, rmax=3).with_(flux="rusanov"), 3, 20),
    (cube_config(nx=4, ny=5, nz=3, G=3, rmax=8).with_(flux="central"), 8, 60),
]


@pytest.mark.parametrize("case", range(len(WORKLOADS)))
def test_transport_sum_of_fp32_cores_is_the_rounded_fp64_one(tt, case):
    wl, r, cap = WORKLOADS[case]
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, wl)
    a = random_tt(plan.n, [r, min(r, plan.n[2])], seed=case)
    rows = a[0].shape[1]
    a[0] = a[0] * (10.0 ** np.linspace(2, -40, rows))[None, :, None]
    a = [c.astype(np.float32).astype(np.float64) for c in a]
    core = []
    for dtype in ("f32", "f64"):
        x = tt.TT.from_cores(a, rcap=[r, r], dtype=dtype)
        out = tt.TT(plan.n, [cap, cap], dtype)
        tt.tt_apply_transport(ctx, plan, x, out)
        ctx.sync()
        core.append(np.asarray(out.to_cores()[0], dtype=np.float64))
    got, want = core
    assert np.all(np.abs(got - want) <= 2.0 ** -23 * np.abs(want) + 2.0 ** -149)
    assert np.any(want != 0.0)
