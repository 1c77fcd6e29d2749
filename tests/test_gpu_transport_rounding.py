"""The FP32 materialised transport sum, formed in pairs of FP32 numbers, is the FP64 one rounded once: an error of
2^-46 turns a rounding at most once in some 2^22 entries, and over 67 million no bit differs."""
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


@pytest.mark.parametrize("flux", ["upwind", "central"])
def test_every_bit_of_the_rounded_sum(tt, flux):
    wl = plane_config1(nx=128, ny=128, G=64, ntheta=4, nphi=8, rmax=16).with_(flux=flux)
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, wl)
    z = torch.randn(wl.nrow, 16, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    ncol = 16 * (5 if flux == "upwind" else 3)
    core = []
    for dtype in ("f32", "f64"):
        x, out = tt.TT(plan.n, [16, 8], dtype), tt.TT(plan.n, [ncol, 40], dtype)
        x.cores[0].copy_(z)
        x.rank.copy_(torch.tensor([1, 16, 8, 1], dtype=torch.int32))
        tt.tt_apply_transport(ctx, plan, x, out)
        ctx.sync()
        core.append(out.cores[0])
    assert core[0].abs().max() > 0
    assert int((core[0] != core[1].float()).sum()) == 0


@pytest.mark.parametrize("flux", ["upwind", "central", "rusanov"])
@pytest.mark.parametrize("dt", [1e-25, 1e-32, 1e-42])
def test_coefficients_near_the_end_of_the_fp32_numbers(tt, dt, flux):
    # entries of a size that keeps the products in range
    wl = plane_config1(nx=16, ny=12, G=8, ntheta=4, nphi=8, rmax=8).with_(flux=flux, dt=dt)
    ctx = tt.Context(0)
    plan = tt.Plan(ctx, wl)
    z = 1e20 * torch.randn(wl.nrow, 8, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    core = []
    for dtype in ("f32", "f64"):
        x, out = tt.TT(plan.n, [8, 8], dtype), tt.TT(plan.n, [72, 72], dtype)
        x.cores[0].copy_(z)
        x.rank.copy_(torch.tensor([1, 8, 8, 1], dtype=torch.int32))
        tt.tt_apply_transport(ctx, plan, x, out)
        ctx.sync()
        core.append(out.cores[0])
    assert core[0][:, 8:].abs().max() > 0
    assert int((core[0] != core[1].float()).sum()) == 0
