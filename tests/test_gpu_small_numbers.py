"""Entries at the lower end of FP32 storage.  Rows down to 2^-112 keep their own accuracy through the FP32 update
(1e-5 of the row, as rows of every size), and FP64 passes over FP32 storage keep its subnormal numbers: columns
below 2^-126 whose right parts scale them back (1e-5, FP32 storage)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import naive_tt as nt  # noqa: E402
from paper_2602_00290_gb300.workloads import random_tt  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


@pytest.mark.parametrize("rows,rank", [(1024, 9), (1153, 32), (1100, 50)])
@pytest.mark.parametrize("prec", ["mixed", "mixed_3xtf32", "fp64"])
def test_small_rows_keep_their_accuracy(tt, rows, rank, prec):
    a = random_tt([rows, 70], [rank], seed=rows + rank)
    a[0] = a[0] * (2.0 ** -(113.0 * np.arange(rows) / rows).astype(int))[None, :, None]
    a = [c.astype(np.float32).astype(np.float64) for c in a]
    x = tt.TT.from_cores(a, dtype="f32")
    ctx = tt.Context(0)
    tt.tt_round(ctx, x, 0.0, rank, prec)
    ctx.sync()
    got, want = nt.full(x.to_cores()), nt.full(a)
    assert (np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)).max() < 1e-5


@pytest.mark.parametrize("rows", [60, 300, 5000])
def test_fp64_passes_keep_subnormal_columns(tt, rows):
    a = random_tt([rows, 70], [9], seed=rows)
    scale = np.where(np.arange(9) < 5, 1.0, 2.0 ** -133)
    right = np.where(np.arange(9) < 5, 1.0, 2.0 ** 122)  # 2^-11 of the other columns
    a = [a[0] * scale[None, None, :], a[1] * right[:, None, None]]
    a = [c.astype(np.float32).astype(np.float64) for c in a]
    x = tt.TT.from_cores(a, dtype="f32")
    ctx = tt.Context(0)
    tt.tt_round(ctx, x, 0.0, 9, "fp64")
    ctx.sync()
    got, want = nt.full(x.to_cores()), nt.full(a)
    assert np.linalg.norm(got - want) < 1e-5 * np.linalg.norm(want)
    # the small columns by themselves: their part of the tensor, to the storage's rounding of the whole
    part = a[0][0][:, 5:] @ a[1][5:, :, 0]
    assert np.linalg.norm((got - want)) < 1e-2 * np.linalg.norm(part)
