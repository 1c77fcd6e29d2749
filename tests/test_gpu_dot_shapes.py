"""Inner products whose column counts lie outside the exact products' plans, after ones that lie inside, and in
several passes of rows with enough columns for the exact form: 1e-12 of the norms, as every inner product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_00290_gb300.workloads import random_tt  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def inner(p, q):
    return float(np.sum((p[0][0].T @ q[0][0]) * (p[1][:, :, 0] @ q[1][:, :, 0].T)))


@pytest.mark.parametrize("pairs,rows,dtype", [
    ([(2, 5), (1, 1005)], 16384, "f64"),
    ([(3, 256), (2, 1256)], 16390, "f32"),
    ([(20, 20)], (1 << 18) + 77, "f64"),
    ([(7, 6), (2, 3), (1, 40)], (1 << 18) + 77, "f32"),
    ([(9, 8), (2, 3), (1, 40)], (1 << 18) + 77, "f64"),
    ([(1, 140)], 1 << 18, "f64"),
])
def test_dots_in_turn(tt, pairs, rows, dtype):
    ctx = tt.Context(0)
    for rx, ry in pairs:
        a, b = random_tt([rows, 8], [rx], seed=rx), random_tt([rows, 8], [ry], seed=ry + 1)
        if dtype == "f32":
            a, b = ([c.astype(np.float32).astype(np.float64) for c in t] for t in (a, b))
        x, y = tt.TT.from_cores(a, dtype=dtype), tt.TT.from_cores(b, dtype=dtype)
        for u, v, p, q in ((x, y, a, b), (y, x, b, a), (x, x, a, a)):
            norms = (inner(p, p) * inner(q, q)) ** 0.5
            assert abs(tt.tt_dot(ctx, u, v).item() - inner(p, q)) <= 1e-12 * norms


def launches(tt, rows, rx, ry, dtype):
    x, y = (tt.TT.from_cores(random_tt([rows, 8], [r], seed=r), dtype=dtype) for r in (rx, ry))
    ctx = tt.Context(0)
    ctx.counters(reset=True)
    tt.tt_dot(ctx, x, y)
    return sum(ctx.counters()[1].values())


@pytest.mark.parametrize("rows,rx,ry,dtype,exact", [
    (1000, 32, 32, "f64", False), (16384, 2, 3, "f64", True), (1 << 18, 2, 3, "f64", True), (1 << 18, 1, 140, "f64", False),
    ((1 << 18) + 1, 2, 3, "f64", False), ((1 << 18) + 1, 15, 15, "f64", False), ((1 << 18) + 1, 16, 16, "f64", True),
    ((1 << 18) + 1, 5, 5, "f32", False), ((1 << 18) + 1, 6, 6, "f32", True), ((1 << 18) + 1, 2, 32, "f32", False),
])
def test_narrow_products_of_many_rows_take_the_sums(tt, rows, rx, ry, dtype, exact):
    # the exact form is several launches more; where it took longer than the sums, the sums stay
    assert (launches(tt, rows, rx, ry, dtype) > launches(tt, 1000, rx, ry, dtype)) == exact
