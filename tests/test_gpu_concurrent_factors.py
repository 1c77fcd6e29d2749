"""Triangular factors of more than 32 columns (a cluster of CTAs that write each other's shared memory) started
while other streams keep the SMs busy, so that the CTAs of a cluster come up at different times: every
rounding returns the bits of the same rounding alone."""
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


@pytest.mark.parametrize("rank", [33, 65, 97, 120])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_factors_on_a_busy_device(tt, rank, prec):
    # a factor is a few kernels: many roundings in flight on streams of their own beside long-running products
    cores = random_tt([513, 130], [rank], seed=rank)
    alone = tt.TT.from_cores(cores, rcap=[rank])
    ctx = tt.Context(0)
    tt.tt_round(ctx, alone, 0.0, rank, prec)
    ctx.sync()
    want = alone.to_cores()
    streams = [torch.cuda.Stream() for _ in range(12)]
    lanes = [(tt.Context(0, stream=s), tt.TT.from_cores(cores, rcap=[rank])) for s in streams]
    busy = torch.cuda.Stream()
    a = torch.randn(2048, 2048, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        for _ in range(8):
            a = (a @ a) * 1e-2
    for c, x in lanes:
        tt.tt_round(c, x, 0.0, rank, prec)
    torch.cuda.synchronize()
    for c, x in lanes:
        c.sync()
        got = x.to_cores()
        assert all((p == q).all() for p, q in zip(got, want))
