"""The kernels of the materialised transport sum, chosen by entries, columns and rows, give the same numbers: an output of
larger capacity takes another kernel for the same state.  They form an entry by the same operations (FP64, or pairs
of FP32 numbers), so the live columns are equal bit by bit and the others zero."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_00290_gb300.workloads import plane_config1  # noqa: E402


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


# cells, groups, rank and output capacities
SHAPES = [(13, 11, 7, 3, (30, 200, 300)),       # 1,001 rows
          (31, 17, 4, 8, (72, 130, 255)),       # 2,108 rows
          (41, 37, 11, 5, (45, 100, 256)),      # 16,687 rows
          (61, 59, 10, 4, (36, 100, 255))]      # 35,990 rows: 64 a CTA in FP32


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("flux,faces", [("upwind", None), ("upwind", (0.9, None, 0.6, None, None, 0.7)),
                                        ("central", None), ("rusanov", None)])
def test_every_kernel_gives_the_same_columns(tt, flux, faces, dtype, shape):
    nx, ny, groups, r, caps = shape
    wl = plane_config1(nx=nx, ny=ny, G=groups, ntheta=4, nphi=8, rmax=r).with_(flux=flux)
    if faces:
        wl = wl.with_(inflow_temperature=faces)
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, wl)
    x = tt.TT(plan.n, [r, r], dtype)
    x.cores[0].copy_(torch.randn(wl.nrow, r, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda"))
    x.rank.copy_(torch.tensor([1, r, r, 1], dtype=torch.int32))
    live, cores = 0, []
    for cap in caps:
        out = tt.TT(plan.n, [cap, cap], dtype)
        out.cores[0].fill_(float("nan"))
        tt.tt_apply_transport(ctx, plan, x, out)
        ctx.sync()
        live = int(out.rank[1])
        cores.append(out.cores[0].view(wl.nrow, cap))
    assert r < live <= caps[0]
    for c in cores:
        assert int((c[:, :live] != cores[0][:, :live]).sum()) == 0
        assert int((c[:, live:] != 0).sum()) == 0
