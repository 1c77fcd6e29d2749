"""FP64 updates of narrow passes from digits (1,024 rows and more) keep the accuracy of the FP64 FMA update (fewer
rows).  The angular core holds unit vectors, so that the pass's weights are the new angular core itself, and its
products are formed again in extended precision: an FMA sum of n terms rounds n times, the digits once, so the
root mean square of the rounding against sum |z||w| is no larger (a tenth for the scatter)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = 512


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


@pytest.mark.parametrize("rank", [2, 5, 9, 17, 32])
def test_digits_are_as_exact_as_fp64_sums(tt, rank):
    ctx = tt.Context(0)
    unit = np.eye(rank, 40).reshape(rank, 40, 1)
    square = [0.0, 0.0]
    for seed in range(4):
        rng = np.random.default_rng(100 * rank + seed)
        z = rng.standard_normal((ROWS, rank)) * 0.7 ** np.arange(rank)[None, :]
        for i, copies in enumerate((1, 3)):
            x = tt.TT.from_cores([np.tile(z, (copies, 1))[None], unit])
            tt.tt_round(ctx, x, 0.0, rank)
            ctx.sync()
            got, right = (c[..., 0] if c.shape[2] == 1 else c[0] for c in x.to_cores())
            w = right[:, :rank].T
            want = z.astype(np.longdouble) @ w.astype(np.longdouble)
            d = (got[:ROWS] - want) / (np.abs(z) @ np.abs(w))
            square[i] += float((d * d).mean())
    assert square[1] ** 0.5 <= 1.1 * square[0] ** 0.5, (square[1] / square[0]) ** 0.5
