"""Workloads of the tensor-train transport library, each as one pass through its public entry points.

A case is a plain dict; ``prepare`` makes what a program holds between passes (a context, plans, a
checkpointed state), ``run`` makes one pass and returns what a program reads from it, ``exact``
gives the same numbers from plain torch in 64 bits, and ``work`` counts what a pass cannot do
without.

A step case restores its state from a checkpoint and steps once, so every pass does the same work.
The cores of a rounded state are unique only up to a gauge (signs and rotations between cores), so
a pass returns the physical fields instead of the cores: the energy density of every (cell, group)
row as the library reports it, and either the whole intensity I[row, ordinate] (up to _DENSE
values) or the flux and pressure moments of every row; the energy report and the live ranks beside
them.  What the mixed precisions compute is accurate to FP32 and is returned as FP32.
"""
import math

import numpy as np
import torch

import paper_2602_00290_gb300 as tt
from paper_2602_00290_gb300 import workloads

_DENSE = 1 << 22  # intensities returned whole up to this many values


def listed():
    return [
        # the 1-D verification slab (64 cells, 16 groups, 8 ordinates, exact rank) in FP64: the smallest call
        dict(name="slab_fp64", kind="step", ndim=1, nx=64, ny=1, nz=1, groups=16, ntheta=8, nphi=1, rank=8, tol=0.0,
             precision="fp64", storage="f64", flux="upwind", inflow=False, rounding="tsqr", graphs=True),
        # the Gaussian-diffusion slab (128 cells, 8 groups, 16 ordinates, central flux): thousands of tiny steps
        dict(name="slab_diffusion_mixed", kind="step", ndim=1, nx=128, ny=1, nz=1, groups=8, ntheta=16, nphi=1,
             rank=12, tol=1e-6, precision="mixed", storage="f32", flux="central", inflow=False, rounding="tsqr",
             graphs=True),
        # a small plane with an inflow face, one of a parameter study, stepped eagerly; odd sizes
        dict(name="plane_small_mixed", kind="step", ndim=2, nx=33, ny=31, nz=1, groups=17, ntheta=8, nphi=16, rank=8,
             tol=1e-6, precision="mixed", storage="f32", flux="upwind", inflow=True, rounding="tsqr", graphs=False),
        # the benchmark plane (128 x 128 cells, 64 groups, 16 x 32 ordinates, r = 32) at its headline precision
        dict(name="plane_3xtf32", kind="step", ndim=2, nx=128, ny=128, nz=1, groups=64, ntheta=16, nphi=32, rank=32,
             tol=1e-6, precision="mixed_3xtf32", storage="f32", flux="upwind", inflow=False, rounding="tsqr",
             graphs=True),
        # the same plane in FP64, the reference precision
        dict(name="plane_fp64", kind="step", ndim=2, nx=128, ny=128, nz=1, groups=64, ntheta=16, nphi=32, rank=32,
             tol=1e-6, precision="fp64", storage="f64", flux="upwind", inflow=False, rounding="tsqr", graphs=True),
        # the largest problem of the batch recipe on its own (192 x 192 cells, 96 groups, r = 48, inflow)
        dict(name="plane_large_mixed", kind="step", ndim=2, nx=192, ny=192, nz=1, groups=96, ntheta=16, nphi=32,
             rank=48, tol=1e-6, precision="mixed", storage="f32", flux="upwind", inflow=True, rounding="tsqr",
             graphs=True),
        # three dimensions with the Rusanov flux, FP64 storage of the state and mixed arithmetic; ragged sizes
        dict(name="cube_rusanov_mixed", kind="step", ndim=3, nx=29, ny=26, nz=23, groups=12, ntheta=8, nphi=16,
             rank=16, tol=1e-6, precision="mixed", storage="f64", flux="rusanov", inflow=False, rounding="tsqr",
             graphs=False),
        # Gram-based rounding in FP64, the cheaper factor for loose tolerances
        dict(name="plane_gram_fp64", kind="step", ndim=2, nx=96, ny=80, nz=1, groups=32, ntheta=8, nphi=16, rank=16,
             tol=1e-3, precision="fp64", storage="f64", flux="upwind", inflow=False, rounding="gram", graphs=True),
        # a linear combination of two solutions (axpy) recompressed (round) in FP64
        dict(name="combine_fp64", kind="combine", ndim=2, nx=48, ny=48, nz=1, groups=32, ntheta=8, nphi=16, rank=20,
             tol=1e-5, precision="fp64", storage="f64"),
        # the materialised transport sum of a state, for analysis outside the fused step
        dict(name="transport_f32", kind="transport", ndim=2, nx=128, ny=128, nz=1, groups=64, ntheta=16, nphi=32,
             rank=16, storage="f32", flux="upwind", inflow=True),
        # the distance of two solutions from three inner products
        dict(name="distance_fp64", kind="distance", ndim=2, nx=128, ny=128, nz=1, groups=64, ntheta=16, nphi=32,
             rank=32, storage="f64"),
        # independent problems of uneven shape stepped together (the batch recipe with cells and groups halved)
        dict(name="batch_mixed", kind="batch", problems=32, scale=2, recipe=3, tol=1e-6, precision="mixed",
             storage="f32"),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 6 + ["combine", "transport", "distance", "batch"])
    if kind == "batch":
        return dict(kind="batch", problems=rng.randint(4, 32), scale=rng.choice([2, 3, 4]), recipe=rng.randint(1, 99),
                    tol=1e-6, precision=rng.choice(["mixed", "mixed_3xtf32"]), storage="f32")
    ntheta, nphi = rng.choice([(8, 16), (12, 24), (16, 32)])
    case = dict(kind=kind, ndim=2, nx=log(12, 160), ny=log(12, 160), nz=1, groups=log(4, 96), ntheta=ntheta,
                nphi=nphi, rank=rng.randint(4, 32))
    if kind == "combine":
        return dict(case, nx=log(8, 64), ny=log(8, 64), groups=log(4, 32), rank=rng.randint(4, 20), tol=1e-5,
                    precision="fp64", storage="f64")
    if kind == "distance":
        return dict(case, storage=rng.choice(["f32", "f64"]))
    if kind == "transport":
        return dict(case, rank=rng.randint(3, 20), storage=rng.choice(["f32", "f64"]),
                    flux=rng.choice(["upwind", "rusanov"]), inflow=False)
    ndim = rng.choice([1, 2, 2, 2, 3])
    flux = rng.choice(["upwind", "upwind", "rusanov", "central"])
    if ndim == 1:
        case.update(ndim=1, nx=log(48, 512), ny=1, groups=log(4, 64), ntheta=rng.choice([8, 16, 24]), nphi=1)
        case["rank"] = rng.randint(4, case["ntheta"] - 2)
    elif ndim == 3:
        case.update(ndim=3, nx=log(6, 32), ny=log(6, 32), nz=log(6, 32), groups=log(4, 16), ntheta=8, nphi=16,
                    rank=rng.randint(4, 16))
    prec = rng.choice(["fp64", "mixed", "mixed_3xtf32"])
    return dict(case, tol=1e-6, precision=prec, storage="f64" if prec == "fp64" else rng.choice(["f32", "f32", "f64"]),
                flux=flux, inflow=flux == "upwind" and rng.random() < 0.4, rounding="tsqr",
                graphs=rng.random() < 0.7)


# --- inputs ---------------------------------------------------------------------------------------

def _workload(case, seed):
    rank, tol = case["rank"], case.get("tol", 1e-6)
    size = dict(nx=case["nx"], G=case["groups"], ntheta=case["ntheta"], rmax=rank, tol=tol)
    if case["ndim"] == 1 and case.get("flux") == "central":
        wl = workloads.gaussian_diffusion_config(seed=seed, **size)
    elif case["ndim"] == 1:
        nx, groups = case["nx"], case["groups"]
        edges = workloads.group_edges(groups)
        ka = workloads.opacity_rows(np.ones(nx), edges, workloads.line_factors(groups, seed=seed))
        wl = workloads.slab_config0().with_(
            nx=nx, ngroup=groups, ntheta=case["ntheta"], dt=0.64 / nx, group_edges=edges,
            temperature=workloads.linear_temperature(nx), rho_kappa_a=ka, rho_kappa_s=0.1 * ka, tol=tol, rmax=rank)
    elif case["ndim"] == 2:
        wl = workloads.plane_config1(ny=case["ny"], nphi=case["nphi"], seed=seed, cfl=0.4, **size)
        wl = wl.with_(dt=0.4 / max(case["nx"], case["ny"]))
    else:
        wl = workloads.cube_config(ny=case["ny"], nz=case["nz"], nphi=case["nphi"], seed=seed, **size)
    wl = wl.with_(flux=case.get("flux", "upwind"))
    return wl.with_(inflow_temperature=(0.7,) + (None,) * 5) if case.get("inflow") else wl


def _cores(wl, rank, seed, dtype):
    """A state in mid-run as cores on the GPU: the merged core's columns are smooth modes over the
    cells on a Planck-like spectrum with a little cell-to-cell variation, graded like the singular
    values of a solution (the first column positive), and the angular cores have orthonormal rows."""
    gen = torch.Generator(device="cuda").manual_seed(2 * seed + 1)
    f64 = dict(dtype=torch.float64, device="cuda")

    def rand(*shape):
        return torch.rand(*shape, generator=gen, **f64)

    x = torch.arange(wl.nx, **f64) / wl.nx
    y = torch.arange(wl.ny, **f64) / wl.ny
    z = torch.arange(wl.nz, **f64) / wl.nz
    wave = 12.0 * rand(3, rank)
    phase = 6.283 * rand(3, rank)
    cell = (torch.cos(z[:, None] * wave[2] + phase[2])[:, None, None]
            * torch.cos(y[:, None] * wave[1] + phase[1])[None, :, None]
            * torch.cos(x[:, None] * wave[0] + phase[0])[None, None, :])
    cell = cell.reshape(wl.ncell, rank)
    cell[:, 0] = 1.5 + cell[:, 0]
    nu = torch.as_tensor(workloads.representative_nu(wl.group_edges), **f64).clamp(1e-3, 40.0)
    temp = 0.5 + 0.5 * rand(1, rank)
    spectrum = nu[:, None] ** 3 / torch.expm1(nu[:, None] / temp) + 1e-6
    Z = (cell[:, None, :] * spectrum[None]).reshape(wl.nrow, rank)
    Z *= 1.0 + 0.02 * torch.randn(wl.nrow, rank, generator=gen, **f64)
    Z *= 0.6 ** torch.arange(rank, **f64)
    small = [wl.ntheta] + ([wl.nphi] if wl.ndim > 1 else [])
    cores = [Z]
    if len(small) == 1:
        q = torch.linalg.qr(torch.randn(small[0], rank, generator=gen, **f64)).Q
        cores.append(q.T.reshape(rank * small[0], 1))
    else:
        r2 = min(rank, small[1])
        mid = torch.randn(rank, small[0], r2, generator=gen, **f64) * 0.8 ** torch.arange(r2, **f64)
        mid = torch.linalg.qr(mid.reshape(rank, small[0] * r2).T).Q.T if rank <= small[0] * r2 else mid
        last = torch.linalg.qr(torch.randn(small[1], r2, generator=gen, **f64)).Q.T
        cores += [mid.reshape(rank, small[0], r2), last.reshape(r2, small[1])]
    return [c.to(torch.float32).double() if dtype == "f32" else c for c in cores]


def _state(n, cores, rcap, dtype):
    """The cores (first [N, r], middle [r, n1, r2], last) in the library's capacity layout."""
    x = tt.TT(n, rcap, dtype)
    rank = cores[0].shape[1]
    x.cores[0][:, :rank] = cores[0]
    if len(n) == 2:
        x.cores[1].view(x.rcap[1], n[1])[:rank] = cores[1].reshape(rank, n[1])
        live = [1, rank, 1]
    else:
        r2 = cores[2].shape[0]
        x.cores[1].view(x.rcap[1], n[1], x.rcap[2])[:rank, :, :r2] = cores[1]
        x.cores[2].view(x.rcap[2], n[2])[:r2] = cores[2]
        live = [1, rank, r2, 1]
    x.rank.copy_(torch.tensor(live, dtype=torch.int32))
    return x


def _modes(wl):
    return [wl.nrow, wl.ntheta] + ([wl.nphi] if wl.ndim > 1 else [])


def _buffers(x):
    return list(x.cores) + [x.rank]


def _angles(wl):
    """Solid angles and direction cosines over the flattened ordinates."""
    if wl.ndim == 1:
        mu, w = np.polynomial.legendre.leggauss(wl.ntheta)
        return 2.0 * np.pi * w, mu[None, :]
    mu = -1.0 + (2.0 * np.arange(wl.ntheta) + 1.0) / wl.ntheta
    phi = (2.0 * np.arange(wl.nphi) + 1.0) * np.pi / wl.nphi
    st = np.sqrt(1.0 - mu * mu)
    n = np.stack([np.outer(st, np.cos(phi)), np.outer(st, np.sin(phi)), np.outer(mu, np.ones(wl.nphi))])
    return np.full(wl.nangle, 4.0 * np.pi / wl.nangle), n.reshape(3, -1)[:wl.ndim]


def _moments(wl, dtype):
    """Columns dOmega n_a and dOmega n_a n_b (flux and pressure) over the ordinates."""
    dom, n = _angles(wl)
    cols = [dom * v for v in n] + [dom * n[a] * n[b] for a in range(len(n)) for b in range(a, len(n))]
    return torch.as_tensor(np.stack(cols, axis=1), dtype=dtype, device="cuda")


def prepare(case, seed):
    tt.lib()
    ctx = tt.Context(0)
    state = dict(case=dict(case), ctx=ctx)
    if case["kind"] == "batch":
        wls = _batch(case)
        plans = [tt.Plan(ctx, wl) for wl in wls]
        start = [_state(p.n, _cores(wl, wl.rmax, seed + i, case["storage"]), [wl.rmax] * 2, case["storage"])
                 for i, (p, wl) in enumerate(zip(plans, wls))]
        live = [p.new_state([wl.rmax] * 2, case["storage"]) for p, wl in zip(plans, wls)]
        state.update(wls=wls, plans=plans, start=[b for x in start for b in _buffers(x)],
                     live=[b for x in live for b in _buffers(x)], states=live,
                     batch=tt.Batch(ctx, plans, live, case["tol"], [wl.rmax for wl in wls], case["precision"]))
        return state
    wl = _workload(case, seed)
    n, rank, dtype = _modes(wl), case["rank"], case["storage"]
    caps = [rank] * (len(n) - 1)
    x0 = _state(n, _cores(wl, rank, seed, dtype), caps, dtype)
    state.update(wl=wl)
    if case["kind"] == "distance":
        state.update(x=x0, y=_state(n, _cores(wl, rank, seed + 7, dtype), caps, dtype))
        return state
    if case["kind"] == "combine":
        caps = [2 * c for c in caps]
        y0 = _state(n, _cores(wl, rank, seed + 7, dtype), caps, dtype)
        y = tt.TT(n, caps, dtype)
        state.update(x=x0, y=y, start=_buffers(y0), live=_buffers(y))
        return state
    plan = tt.Plan(ctx, wl)
    state.update(plan=plan)
    if case["kind"] == "transport":
        blocks = 1 + 2 * wl.ndim
        state.update(x=x0, out=tt.TT(n, [blocks * rank + int(case["inflow"])] * (len(n) - 1), dtype))
        return state
    ctx.set_rounding(case["rounding"])
    ctx.set_graphs(case["graphs"])
    x = tt.TT(n, caps, dtype)
    state.update(x=x, start=_buffers(x0), live=_buffers(x), moments=_moments(wl, x.cores[0].dtype),
                 energy=torch.zeros(4, dtype=torch.float64, device="cuda"))
    return state


def _batch(case):
    return workloads.batch_config3(nprob=case["problems"], seed=case["recipe"], scale=case["scale"], tol=case["tol"])


# --- passes ---------------------------------------------------------------------------------------

def _result(v, case):
    return v if case.get("precision", "fp64") == "fp64" else v.float()


def _right(x):
    """Right part [rcap_1, ordinates] of a state."""
    if x.d == 2:
        return x.cores[1].view(x.rcap[1], x.n[1])
    mid = x.cores[1].view(x.rcap[1] * x.n[1], x.rcap[2])
    return (mid @ x.cores[2].view(x.rcap[2], x.n[2])).view(x.rcap[1], -1)


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "batch":
        torch._foreach_copy_(state["live"], state["start"])
        state["batch"].step(1)
        energy = [tt.tt_energy_density(ctx, p, x) for p, x in zip(state["plans"], state["states"])]
        return dict(energy_density=_result(torch.cat(energy), case), ranks=torch.cat([x.rank for x in state["states"]]))
    if kind == "distance":
        x, y = state["x"], state["y"]
        return dict(xx=tt.tt_dot(ctx, x, x), xy=tt.tt_dot(ctx, x, y), yy=tt.tt_dot(ctx, y, y))
    if kind == "transport":
        out = state["out"]
        tt.tt_apply_transport(ctx, state["plan"], state["x"], out)
        return dict(cores=out.cores, ranks=out.rank)
    torch._foreach_copy_(state["live"], state["start"])
    if kind == "combine":
        y = state["y"]
        tt.tt_axpy(ctx, -0.75, state["x"], y)
        tt.tt_round(ctx, y, case["tol"], 2 * case["rank"], case["precision"])
        return dict(intensity=y.cores[0] @ _right(y), ranks=y.rank)
    x = state["x"]
    tt.tt_step(ctx, state["plan"], x, case["tol"], case["rank"], case["precision"], state["energy"])
    out = dict(energy_density=_result(tt.tt_energy_density(ctx, state["plan"], x), case),
               report=_result(state["energy"], case), ranks=x.rank)
    right = _right(x)
    if x.n[0] * right.shape[1] <= _DENSE:
        out["intensity"] = _result(x.cores[0] @ right, case)
    else:
        out["moments"] = _result(x.cores[0] @ (right @ state["moments"]), case)
    return out


def work(case):
    """Bytes of the states and fields read and written once; the products of a rounding: the
    symmetric Gram (or triangular factor) of the summed columns and the projection on the new frame."""
    if case["kind"] == "batch":
        wls = _batch(case)
        per = [_step_work(wl.nrow, wl.nangle, wl.ndim, wl.rmax, wl.rmax, 1, 4, "upwind") for wl in wls]
        return dict(bytes=sum(b for b, _ in per), flops=sum(f for _, f in per))
    rows = case["nx"] * case["ny"] * case["nz"] * case["groups"]
    r, s = case["rank"], 8 if case["storage"] == "f64" else 4
    if case["kind"] == "distance":
        return dict(bytes=2 * rows * r * s, flops=2 * rows * (r * r + r * (r + 1)))
    if case["kind"] == "transport":
        cols = (1 + 2 * case["ndim"]) * r + int(case["inflow"])
        return dict(bytes=rows * s * (r + cols), flops=2 * rows * (cols - r))
    if case["kind"] == "combine":
        b, f = rows * s * 3 * r, rows * (4 * r * r + 2 * 2 * r * 2 * r)
        return dict(bytes=b + 8 * rows * case["ntheta"] * case["nphi"], flops=f)
    b, f = _step_work(rows, case["ntheta"] * case["nphi"], case["ndim"], r, min(r, case["nphi"]), int(case["inflow"]),
                      s, case["flux"])
    return dict(bytes=b, flops=f)


def _step_work(rows, nang, ndim, r, r2, nbc, s, flux):
    c1 = (1 + ndim * (1 if flux == "central" else 2)) * r + nbc
    c2 = r + 1
    flops = rows * (c1 * c1 + 2 * c1 * r + c2 * c2 + 2 * c2 * r) + 2 * nang * c1 * c1
    # the state in and out, opacities and emission in, the energy density out
    return rows * (2 * r * s + 3 * 8 + 8), flops


# --- the same numbers in 64 bits ------------------------------------------------------------------

def _planck_rows(wl):
    """Group emission per merged row: c a T^4 / 4 pi * 15 / pi^4 * int t^3 / (e^t - 1) over the group."""
    temps, inverse = np.unique(np.asarray(wl.temperature, dtype=float), return_inverse=True)
    return torch.as_tensor(_planck(temps, wl)[inverse].reshape(-1), device="cuda")


def _planck(temps, wl):
    node, weight = np.polynomial.legendre.leggauss(32)
    edges = np.asarray(wl.group_edges, dtype=float)
    out = np.zeros((len(temps), wl.ngroup))
    for g in range(wl.ngroup):
        lo = np.minimum(edges[g] / temps, 700.0)
        hi = np.minimum(edges[g + 1] / temps, lo + 60.0)
        cuts = np.linspace(0.0, 1.0, 17)
        for a, b in zip(cuts[:-1], cuts[1:]):
            t0, t1 = lo + a * (hi - lo), lo + b * (hi - lo)
            t = 0.5 * (t1 - t0)[:, None] * node + 0.5 * (t1 + t0)[:, None]
            f = np.where(t > 0, t ** 3 / np.expm1(np.maximum(t, 1e-300)), 0.0)
            out[:, g] += 0.5 * (t1 - t0) * (f @ weight)
    return out * (wl.c * wl.a_rad * temps ** 4 / (4.0 * np.pi) * 15.0 / np.pi ** 4)[:, None]


def _shift(Z, wl, axis, sign):
    """Row k -> Z of the neighbour cell along an axis, zero outside the grid."""
    g = Z.reshape(wl.nz, wl.ny, wl.nx, wl.ngroup, -1)
    dim = 2 - axis
    out = torch.zeros_like(g)
    n = g.shape[dim]
    if sign > 0:
        out.narrow(dim, 0, n - 1).copy_(g.narrow(dim, 1, n - 1))
    else:
        out.narrow(dim, 1, n - 1).copy_(g.narrow(dim, 0, n - 1))
    return out.reshape(Z.shape)


def _terms(wl):
    """(axis, which difference, angular factor on core 1, on core 2) of the transport operators."""
    dom, n = _angles(wl)
    one = np.ones(wl.nphi)
    if wl.ndim == 1:
        full = [(n[0], one)]
    else:
        mu = -1.0 + (2.0 * np.arange(wl.ntheta) + 1.0) / wl.ntheta
        phi = (2.0 * np.arange(wl.nphi) + 1.0) * np.pi / wl.nphi
        st = np.sqrt(1.0 - mu * mu)
        full = [(st, np.cos(phi)), (st, np.sin(phi)), (mu, one)][:wl.ndim]
    out = []
    for a, (f1, f2) in enumerate(full):
        if wl.flux == "upwind":
            for w in (1, -1):
                part = (lambda v: np.where(v >= 0, v, 0.0)) if w > 0 else (lambda v: np.where(v < 0, v, 0.0))
                out.append((a, w, f1, part(f2)) if wl.ndim > 1 and a < 2 else (a, w, part(f1), f2))
        else:
            out.append((a, 2, f1, f2))
            if wl.flux == "rusanov":
                out.append((a, -2, np.ones_like(f1), one))
    return out


def _columns(Z, wl):
    """Columns of the transport sum in rank blocks, and the inflow column of the lower x face."""
    blocks, inflow = [Z], []
    for a, w, _, _ in _terms(wl):
        lam = wl.c * wl.dt / wl.spacing[a]
        lo = _shift(Z, wl, a, -1) if w != -1 else None
        hi = _shift(Z, wl, a, 1) if w != 1 else None
        diff = Z - lo if w == 1 else hi - Z if w == -1 else 0.5 * (hi - lo) if w == 2 else -0.5 * (hi - 2 * Z + lo)
        blocks.append(diff.mul_(-lam))
        if a == 0 and w == 1 and wl.inflow_temperature[0] is not None:
            face = torch.zeros(wl.nz, wl.ny, wl.nx, wl.ngroup, dtype=torch.float64, device="cuda")
            face[:, :, 0] = torch.as_tensor(lam * _planck(np.array([wl.inflow_temperature[0]]), wl)[0], device="cuda")
            inflow.append(face.reshape(-1, 1))
    return torch.cat(blocks + inflow, dim=1)


def _rank_of(sigma, delta, cap):
    tail = torch.sqrt(torch.flip(torch.cumsum(torch.flip(sigma ** 2, [0]), 0), [0])).cpu().numpy()
    k = len(tail)
    if delta is not None:
        k = next((j for j in range(1, len(tail)) if tail[j] <= delta), len(tail))
    return max(1, min(k, cap))


def _round(A, B, modes, tol, cap):
    """SVD rounding of A B (A: rows x c, B: c x ordinates): the new first core and right part."""
    live = A.abs().amax(0) > 0
    Y = torch.linalg.qr(A[:, live], mode="r").R @ B[live]
    norm = torch.linalg.norm(Y)
    delta = None if tol == 0.0 else float(tol * norm / math.sqrt(len(modes)))
    if len(modes) == 2:
        _, s, vh = torch.linalg.svd(Y.reshape(-1, modes[1]), full_matrices=False)
        v2 = vh[:_rank_of(s, delta, cap)].T
        Y2 = (Y.reshape(-1, modes[1]) @ v2).reshape(Y.shape[0], -1)
        _, s, vh = torch.linalg.svd(Y2, full_matrices=False)
        v1 = vh[:_rank_of(s, delta, cap)]
        Bn = (v1.reshape(-1, v2.shape[1]) @ v2.T).reshape(v1.shape[0], -1)
    else:
        _, s, vh = torch.linalg.svd(Y, full_matrices=False)
        Bn = vh[:_rank_of(s, delta, cap)]
    return A @ (B @ Bn.T), Bn


def _full_right(cores, wl):
    if wl.ndim == 1:
        return cores[1].reshape(-1, wl.ntheta)
    return (cores[1].reshape(-1, cores[1].shape[2]) @ cores[2]).reshape(cores[1].shape[0], -1)


def _exact_step(wl, cores):
    """One step: (row emission and coefficients, Z, B after it, energy report)."""
    modes = _modes(wl)[1:]
    Z, B = cores[0], _full_right(cores, wl)
    dom = torch.as_tensor(_angles(wl)[0], device="cuda")
    scale = 4.0 * math.pi / wl.c * float(np.prod(np.asarray(wl.spacing)[:wl.ndim]))
    before = scale * float((Z @ (B @ dom)).sum()) / (4.0 * math.pi)
    rights, factors = [B], []
    for a, w, f1, f2 in _terms(wl):
        f = torch.as_tensor(np.outer(f1, f2).reshape(1, -1), device="cuda")
        rights.append(B * f)
        if a == 0 and w == 1 and wl.inflow_temperature[0] is not None:
            factors.append(f)
    Z, B = _round(_columns(Z, wl), torch.cat(rights + factors), modes, wl.tol, wl.rmax)
    a = wl.c * wl.dt * torch.as_tensor(wl.rho_kappa_a, device="cuda")
    s = wl.c * wl.dt * torch.as_tensor(wl.rho_kappa_s, device="cuda")
    eps = _planck_rows(wl)
    js = Z @ (B @ dom) / (4.0 * math.pi)
    jn = (js + a * eps) / (1.0 + a)
    d = 1.0 / (1.0 + a + s)
    A = torch.cat([d[:, None] * Z, ((a * eps + s * jn) * d)[:, None]], dim=1)
    Z, B = _round(A, torch.cat([B, torch.ones_like(B[:1])]), modes, wl.tol, wl.rmax)
    J = Z @ (B @ dom) / (4.0 * math.pi)
    report = torch.tensor([before, scale * float(J.sum()), scale * float(js.sum()),
                           scale * float((a * (eps - jn)).sum())], dtype=torch.float64, device="cuda")
    return Z, B, 4.0 * math.pi / wl.c * J, report


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = [_exact_step(wl, _cores(wl, wl.rmax, seed + i, case["storage"]))[2]
               for i, wl in enumerate(_batch(case))]
        return dict(energy_density=torch.cat(out), ranks=None)
    wl = _workload(case, seed)
    cores = _cores(wl, case["rank"], seed, case["storage"])
    if kind in ("distance", "combine"):
        other = _cores(wl, case["rank"], seed + 7, case["storage"])
        B, Bo = _full_right(cores, wl), _full_right(other, wl)
        if kind == "combine":
            A = torch.cat([other[0], -0.75 * cores[0]], dim=1)
            Z, Bn = _round(A, torch.cat([Bo, B]), _modes(wl)[1:], case["tol"], 2 * case["rank"])
            return dict(intensity=Z @ Bn, ranks=None)
        dots = [((p[0].T @ q[0]) * (u @ v.T)).sum().reshape(1)
                for p, u, q, v in ((cores, B, cores, B), (cores, B, other, Bo), (other, Bo, other, Bo))]
        return dict(xx=dots[0], xy=dots[1], yy=dots[2])
    if kind == "transport":
        return dict(cores=_exact_transport(wl, cores), ranks=None)
    Z, B, E, report = _exact_step(wl, cores)
    out = dict(energy_density=E, report=report, ranks=None)
    if wl.nrow * B.shape[1] <= _DENSE:
        out["intensity"] = Z @ B
    else:
        out["moments"] = Z @ (B @ _moments(wl, torch.float64))
    return out


def _exact_transport(wl, cores):
    """Cores of the transport sum: blocks side by side, block diagonal, stacked."""
    terms = _terms(wl)
    nbc = int(wl.inflow_temperature[0] is not None)
    rank, n1 = cores[0].shape[1], wl.ntheta
    cap = (1 + 2 * wl.ndim) * rank + nbc
    first = torch.zeros(wl.nrow, cap, dtype=torch.float64, device="cuda")
    columns = _columns(cores[0], wl)
    first[:, :columns.shape[1]] = columns
    r2, n2 = cores[2].shape
    mid = torch.zeros(cap, n1, cap, dtype=torch.float64, device="cuda")
    last = torch.zeros(cap, n2, dtype=torch.float64, device="cuda")
    blocks = [(np.ones(n1), np.ones(n2))] + [(f1, f2) for _, _, f1, f2 in terms]
    for t, (f1, f2) in enumerate(blocks):
        mid[t * rank:(t + 1) * rank, :, t * r2:(t + 1) * r2] = cores[1] * torch.as_tensor(f1, device="cuda")[None, :, None]
        last[t * r2:(t + 1) * r2] = cores[2] * torch.as_tensor(f2, device="cuda")
    if nbc:
        mid[len(blocks) * rank, :, len(blocks) * r2] = torch.as_tensor(terms[0][2], device="cuda")
        last[len(blocks) * r2] = torch.as_tensor(terms[0][3], device="cuda")
    return [first, mid.reshape(cap * n1, cap), last.reshape(cap * n2, 1)]
