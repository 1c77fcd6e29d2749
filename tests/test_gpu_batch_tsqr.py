"""The context's TSQR choice reaches a batch that was made before it: the batch steps as one made afterwards, launch
for launch and bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_00290_gb300.workloads import batch_config3  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def make(tt, ctx):
    wls = batch_config3(5, seed=3, scale=8)
    plans = [tt.Plan(ctx, wl) for wl in wls]
    states = [tt.initial_state(p, [w.rmax, w.rmax], "f32") for p, w in zip(plans, wls)]
    return tt.Batch(ctx, plans, states, [w.tol for w in wls], [w.rmax for w in wls], "mixed", nstreams=4), states


@pytest.mark.parametrize("widths,before", [(range(1, 257), 0), (range(1, 257), 1), (range(40, 257), 0), (range(1, 40), 1)])
@pytest.mark.parametrize("variant", ["column", "rowsplit"])
def test_a_choice_made_after_the_batch(tt, widths, before, variant):
    # all passes, the wide ones or the narrow ones alone take the Householder kernels, from the step `before` on
    late, early = tt.Context(0), tt.Context(0)
    b, states = make(tt, late)
    b.step(before)
    for ctx in (late, early):
        for n in widths:
            ctx.set_tsqr("mixed", n, variant, 0)
    want, ref = make(tt, early)
    b.step(3 - before)
    b.sync()
    want.step(3)
    want.sync()
    assert b.info()["launches_per_step"] == want.info()["launches_per_step"]
    for x, y in zip(states, ref):
        p, q = x.to_cores(), y.to_cores()
        # with a step taken before, its round-off is the other factor's
        assert before or all((u == v).all() for u, v in zip(p, q))
        assert x.ranks() == y.ranks() or before
        assert all(np.isfinite(u).all() for u in p)
