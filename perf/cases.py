"""The gas advance's performance cases: what a program that uses this library
has it do, through ``paper_1301_4498_gb300.hydro``, from one small box to a
level of many boxes, in both precisions, with and without the scheme options,
through device and host buffers, alone and with self-gravity, particles and a
refined level.

A pass starts from a snapshot: single steps read state[0] and write state[1]
(``level.cur = 0``); multi-step runs and particle steps first copy the
snapshot back, as a program that restarts from one does.  ``exact`` is a plain
FP64 torch statement of the same scheme on dense arrays.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1301_4498_gb300 import hydro as H
from paper_1301_4498_gb300 import workloads as WL

A0, A1 = 1.0 / 51, 1.0 / 49      # first and last scale factor of a 10-step run
ASTEP = (A1 - A0) / 10
F64 = torch.float64

# Algorithmic operations per zone and step of the advance (+ - x / sqrt one
# each): FP64 arithmetic with the two-shock solver's mean iterations at 1e-10,
# and mixed precision at 1e-6.
FLOPS = {"fp64": 5034, "mixed": 4660}


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # Sod shock tube, FP64, 20 steps in one graph replay: the smallest run
        # of the repository's configurations; launches and latency count
        dict(name="sod_fp64_run20", kind="run", level="sod", n=128, ny=8, precision="fp64",
             steps=20, tune=False),
        # one eager step of one 32^3 box, the plan's defaults: the smallest call
        dict(name="box32_mixed_step", kind="step", level="box", n=32, precision="mixed",
             sigma=0.5, tune=False),
        # one eager step of one 96^3 box in FP64: the plain full-precision form
        dict(name="box96_fp64_step", kind="step", level="box", n=96, precision="fp64",
             sigma=0.5, tune=True),
        # uneven boxes (edges 16..64) of one level, FP64: the batched form
        dict(name="uneven12_fp64_step", kind="step", level="uneven", nbox=12, precision="fp64",
             sigma=0.5, tune=True),
        # uneven boxes, mixed, two steps in one graph replay
        dict(name="uneven48_mixed_run2", kind="run", level="uneven", nbox=48, precision="mixed",
             sigma=0.5, steps=2, tune=True),
        # an eighth of the large batched level: 512 boxes of 32^3 tiling 256^3
        # and 51 boxes of 64^3 at half the cell width, two steps in one replay
        dict(name="level256_mixed_run2", kind="run", level="large", n=256, box=32, nfine=51,
             precision="mixed", sigma=1.0, steps=2, tune=True),
        # one 192^3 box with shock flattening and the second form of the
        # gravity energy source, strong contrasts
        dict(name="box192_flat_mixed_step", kind="step", level="box", n=192, precision="mixed",
             sigma=1.0, flat=True, genergy=1, tune=True),
        # PLM with the linearised solver on ragged boxes (50^3 tiling 100^3)
        dict(name="tiled100_plm_mixed_step", kind="step", level="tiled", n=100, box=50,
             precision="mixed", sigma=0.5, plm=True, linear=True, tune=True),
        # end to end through pinned host buffers, valid cells only
        dict(name="host192_mixed_step", kind="host", level="tiled", n=192, box=64,
             precision="mixed", sigma=1.0, tune=True),
        # self-gravity of a 256^3 level from a cold start
        dict(name="poisson256_mixed", kind="poisson", level="tiled", n=256, box=64,
             precision="mixed", sigma=1.0),
        # one step with gas, one dark-matter particle per cell and self-gravity
        dict(name="cosmo128_mixed_step", kind="cosmo", level="tiled", n=128, box=32,
             precision="mixed", sigma=1.0, tune=True),
        # two coupled levels: 64 boxes of 32^3, 6 of them refined by 2
        dict(name="amr128_mixed_step", kind="amr", level="tiled", n=128, box=32, nfine=6,
             precision="mixed", sigma=1.0, tune=True),
    ]


def _log_even(rng, lo, hi):
    return 2 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2))


def draw(rng):
    """Sizes over the whole ranges (even edges, as the library requires)."""
    kind = rng.choice(["step", "step", "step", "run", "run", "host", "poisson", "cosmo", "amr"])
    sigma = rng.choice([0.5, 1.0])
    tune = rng.random() < 0.7
    if kind in ("step", "run"):
        precision = rng.choice(["mixed", "mixed", "fp64"])
        level = rng.choice(["box", "tiled", "uneven", "large"] if precision == "mixed"
                           else ["box", "tiled", "uneven"])
        c = dict(kind=kind, level=level, precision=precision, sigma=sigma, tune=tune)
        if level == "box":
            c["n"] = _log_even(rng, 16, 200 if precision == "mixed" else 72)
        elif level == "tiled":
            b = 2 * rng.randint(7, 33 if precision == "mixed" else 15)
            c.update(box=b, n=b * rng.randint(2, 4 if precision == "mixed" else 2))
        elif level == "uneven":
            c["nbox"] = rng.randint(2, 48 if precision == "mixed" else 12)
        else:
            c.update(n=128, box=32, nfine=rng.randint(1, 40))
        if kind == "run":
            c["steps"] = rng.randint(1, 4)
        elif precision == "mixed":
            c.update(flat=rng.random() < 0.4, genergy=rng.choice([0, 1]),
                     plm=rng.random() < 0.3, linear=rng.random() < 0.3)
        return c
    if kind == "host":
        b = 2 * rng.randint(12, 32)
        return dict(kind=kind, level="tiled", box=b, n=3 * b, precision="mixed", sigma=sigma,
                    tune=True)
    if kind == "poisson":
        b = rng.choice([16, 24, 32, 48, 64])
        p = rng.choice(["mixed", "mixed", "fp64"])
        return dict(kind=kind, level="tiled", box=b, n=b * rng.choice([2, 4] if b <= 48 else [2]),
                    precision=p, sigma=sigma)
    if kind == "cosmo":
        b = rng.choice([16, 24, 32])
        return dict(kind=kind, level="tiled", box=b, n=b * rng.choice([2, 4]), precision="mixed",
                    sigma=sigma, tune=tune)
    b = 2 * rng.randint(8, 20)
    return dict(kind=kind, level="tiled", box=b, n=4 * b, nfine=rng.randint(1, 6),
                precision="mixed", sigma=sigma, tune=tune)


# ---------------------------------------------------------------- levels and fields
SIZES = (16, 24, 32, 48, 64)


def _parts(case):
    """The level as parts of boxes: (level spec, [(boxes, dense extent
    (nx, ny, nz), dx, bc)...]).  A part is one dense domain whose boxes tile
    it, or several equal single-box domains."""
    lv, n = case["level"], case.get("n")
    if lv == "sod":
        ext = (n, case["ny"], case["ny"])
        spec = WL.single_box_level(*ext, 1.0 / n, (1, 0, 0, 1, 0, 0), name="sod")
        return spec, [([0], ext, 1.0 / n, "sod")]
    if lv == "box":
        return WL.single_box_level(n, n, n, 1.0 / n), [([0], (n, n, n), 1.0 / n, "")]
    if lv == "tiled":
        spec = WL.tiled_level(n, case["box"])
        return spec, [(list(range(spec.nbox)), (n, n, n), 1.0 / n, "")]
    if lv == "uneven":
        ext = np.random.default_rng(3).choice(np.asarray(SIZES), size=(case["nbox"], 3))
        ext = [tuple(int(v) for v in e) for e in ext]
        spec = WL.independent_boxes_level(ext, 1.0 / 128)
        return spec, [([b], e, 1.0 / 128, "") for b, e in enumerate(ext)]
    coarse = WL.tiled_level(n, case["box"])
    fine = WL.independent_boxes_level([(64,) * 3] * case["nfine"], 0.5 / n)
    spec = WL.merge_levels(coarse, fine)
    parts = [(list(range(coarse.nbox)), (n, n, n), 1.0 / n, "")]
    parts += [([coarse.nbox + k], (64,) * 3, 0.5 / n, "") for k in range(case["nfine"])]
    return spec, parts


def _gaussian(ext, count, gen):
    """count unit-variance Gaussian fields with P(k) ~ k^-2, (count, nz, ny, nx)."""
    nx, ny, nz = ext
    dev = "cuda"
    w = torch.randn((count, nz, ny, nx), generator=gen, device=dev, dtype=F64)
    f = torch.fft.rfftn(w, dim=(1, 2, 3))
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device=dev, dtype=F64).view(-1, 1, 1)
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=dev, dtype=F64).view(1, -1, 1)
    kx = torch.arange(nx // 2 + 1, device=dev, dtype=F64).view(1, 1, -1)
    k2 = kz * kz + ky * ky + kx * kx
    k2[0, 0, 0] = 1.0
    amp = 1.0 / k2.sqrt()
    amp[0, 0, 0] = 0.0
    g = torch.fft.irfftn(f * amp, s=(nz, ny, nx), dim=(1, 2, 3))
    return g / g.flatten(1).std(dim=1).view(-1, 1, 1, 1)


def _fields(part, case, gen):
    """Dense conserved state (6, nz, ny, nx) and gravity (3, nz, ny, nx): the
    lognormal comoving field of the repository's workloads (density, k^-2
    velocities, gravity the centred gradient of a Gaussian potential), or the
    Sod tube with a seeded interface position and density."""
    _, ext, dx, what = part
    nx, ny, nz = ext
    if what == "sod":
        r = torch.rand(2, generator=gen, device="cuda", dtype=F64)
        x = (torch.arange(nx, device="cuda", dtype=F64) + 0.5) / nx
        left = x < 0.45 + 0.1 * r[0]
        gm1 = 0.4
        rho = torch.where(left, 1.0 + 0.1 * r[1], 0.125 + 0 * r[1])
        e = torch.where(left, 1.0, 0.1) / gm1
        S = torch.zeros((6, nz, ny, nx), device="cuda", dtype=F64)
        S[0], S[4], S[5] = rho, e, e
        return S, None
    G = _gaussian(ext, 5, gen)
    sg = case["sigma"]
    rho = torch.exp(sg * G[0] - 0.5 * sg * sg)
    rho = rho / rho.mean()
    u = G[1:4]
    u = u * (0.1 / (u * u).sum(0).mean().sqrt())
    phi = G[4]
    g = torch.stack([-(phi.roll(-1, d) - phi.roll(1, d)) for d in (2, 1, 0)])
    g = g * (0.1 / (g * g).sum(0).mean().sqrt())
    re = rho * WL.E0
    S = torch.empty((6, nz, ny, nx), device="cuda", dtype=F64)
    S[0], S[1:4], S[5] = rho, rho * u, re
    S[4] = re + 0.5 * rho * (u * u).sum(0)
    return S, g


def _dense(case, seed):
    """[(dense state, dense gravity)] of every part, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    _, parts = _parts(case)
    return [_fields(p, case, gen) for p in parts]


def _params(case):
    p = dict(precision=case["precision"], gamma=1.4 if case["level"] == "sod" else 5.0 / 3.0,
             cfl=0.5, autotune=int(bool(case.get("tune"))))
    if case.get("genergy"):
        p["grav_energy"] = 1
    if case.get("flat"):
        p["flattening"] = 1
    if case.get("plm"):
        p["reconstruction"] = "plm"
    if case.get("linear"):
        p["riemann_solver"] = "linear"
    return p


def _boxes_of(spec, part):
    """(box, slices of the dense array) for every box of a part."""
    for b in part[0]:
        lo = spec.lo[b] - spec.dom_lo[spec.dom[b]]
        nx, ny, nz = spec.extent(b)
        yield b, (slice(None), slice(lo[2], lo[2] + nz), slice(lo[1], lo[1] + ny),
                  slice(lo[0], lo[0] + nx))


def _view(plan, field, ncomp, b):
    """Valid cells of box b of a level field: a view (ncomp, nz, ny, nx)."""
    off, st = plan.layout_cache[ncomp]
    nx, ny, nz = plan.spec.extent(b)
    blk = field[off[b]:off[b + 1]].view(ncomp, int(st[b]))
    return blk[:, :(nx + 8) * (ny + 8) * (nz + 8)].view(ncomp, nz + 8, ny + 8, nx + 8)[
        :, 4:-4, 4:-4, 4:-4]


def _put(plan, parts, dense, field, ncomp):
    for part, d in zip(parts, dense):
        for b, sl in _boxes_of(plan.spec, part):
            _view(plan, field, ncomp, b).copy_(d[sl])


def _groups(spec):
    """Runs of consecutive boxes of equal extent (their blocks have one stride)."""
    out = []
    for b in range(spec.nbox):
        if out and spec.extent(out[-1][0]) == spec.extent(b):
            out[-1][1] = b + 1
        else:
            out.append([b, b + 1])
    return out


def _views(plan, field, ncomp):
    """Views of every box's valid cells, one per run of equal boxes:
    (boxes, ncomp, nz, ny, nx)."""
    off, st = plan.layout_cache[ncomp]
    out = []
    for b0, b1 in _groups(plan.spec):
        nx, ny, nz = plan.spec.extent(b0)
        blk = field[off[b0]:off[b1]].view(b1 - b0, ncomp, int(st[b0]))
        out.append(blk[:, :, :(nx + 8) * (ny + 8) * (nz + 8)].view(
            b1 - b0, ncomp, nz + 8, ny + 8, nx + 8)[:, :, 4:-4, 4:-4, 4:-4])
    return out


def _cut(spec, parts, dense):
    """Dense arrays of the parts in the layout of _views."""
    per = {}
    for part, d in zip(parts, dense):
        for b, sl in _boxes_of(spec, part):
            per[b] = d[sl]
    return [torch.stack([per[b] for b in range(b0, b1)]) for b0, b1 in _groups(spec)]


def _make(case, dense, with_grav=True, stream=None, spec=None, parts=None, **more):
    if spec is None:
        spec, parts = _parts(case)
    plan = H.Plan(spec, stream=stream, **{**_params(case), **more})
    plan.layout_cache = {c: plan.layout(c) for c in (3, 6)}
    s0, s1 = plan.empty_field(6), plan.empty_field(6)
    _put(plan, parts, [d[0] for d in dense], s0, 6)
    grav = None
    if with_grav and dense[0][1] is not None:
        grav = plan.empty_field(3)
        _put(plan, parts, [d[1] for d in dense], grav, 3)
        plan.fill(grav, 3)
    return plan, H.Level(s0, s1, grav)


def _a(case, steps):
    """Scale factors: fixed at 1 for the tube, else the comoving schedule."""
    if case["level"] == "sod":
        return [1.0] * (steps + 1)
    return [A0 + ASTEP * s for s in range(steps + 1)]


def _particles(n, gen):
    """One particle per cell, displaced up to 0.3 cells, rms velocity 0.1."""
    c = torch.arange(n, device="cuda", dtype=F64) + 0.5
    x = torch.stack(torch.meshgrid(c, c, c, indexing="ij")).reshape(3, -1)
    x = x + 0.3 * (2 * torch.rand(x.shape, generator=gen, device="cuda", dtype=F64) - 1)
    x = torch.remainder(x / n, 1.0).contiguous()
    u = 0.1 * torch.randn(x.shape, generator=gen, device="cuda", dtype=F64)
    m = torch.full((x.shape[1],), 5.0 / x.shape[1], device="cuda", dtype=F64)
    return x, u, m


def _refined(case, spec):
    """The refined coarse boxes: seeded, any neighbourhood."""
    rng = np.random.default_rng(11)
    return sorted(int(b) for b in rng.choice(spec.nbox, size=case["nfine"], replace=False))


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    spec, parts = _parts(case)
    dense = _dense(case, seed)
    st = dict(kind=case["kind"], case=case)
    steps = case.get("steps", 1)
    a = _a(case, steps)
    st["a"] = torch.tensor(a, device="cuda", dtype=F64)
    kind = case["kind"]
    if kind in ("step", "run"):
        plan, lev = _make(case, dense)
        st.update(plan=plan, lev=lev, steps=steps)
        if kind == "run":
            st["snap"] = lev.state[0].clone()
            st["dt"] = torch.zeros(steps + 1, device="cuda", dtype=F64)
            st["out"] = _views(plan, lev.state[steps & 1], 6)
        else:
            st["dt"] = torch.tensor([_cfl(case, parts, dense, a[0])], device="cuda", dtype=F64)
            st["dtn"] = torch.zeros(1, device="cuda", dtype=F64)
            st["out"] = _views(plan, lev.state[1], 6)
    elif kind == "host":
        plan, lev = _make(case, dense)
        packed = torch.cat([v.reshape(-1) for v in _views(plan, lev.state[0], 6)])
        st.update(plan=plan, lev=lev, dt=_cfl(case, parts, dense, a[0]),
                  h_in=torch.empty(packed.numel(), dtype=F64, pin_memory=True),
                  h_out=torch.empty(packed.numel(), dtype=F64, pin_memory=True))
        st["h_in"].copy_(packed)
        st["av"] = a
        lev.state[0].zero_()
    elif kind == "poisson":
        plan, lev = _make(case, dense, with_grav=False)
        ps = H.Poisson(plan, four_pi_G=1.0, precision=case["precision"])
        g = plan.empty_field(3)
        st.update(plan=plan, lev=lev, ps=ps, g=g, out=_views(plan, g, 3))
    elif kind == "cosmo":
        plan, lev = _make(case, dense)
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 7919)
        x, u, m = _particles(case["n"], gen)
        ps = H.Poisson(plan, four_pi_G=1.0, precision=case["precision"])
        rho, gd = ps.dense(1)[0], dense[0][1].contiguous()
        st.update(plan=plan, lev=lev, ps=ps, x0=x, u0=u, m=m, x=x.clone(), u=u.clone(), rho=rho,
                  gd0=gd, gd=gd.clone(), g_new=plan.empty_field(3), av=a,
                  dtv=_cfl(case, parts, dense, a[0]), pdt=torch.zeros(1, device="cuda", dtype=F64),
                  dtn=torch.zeros(1, device="cuda", dtype=F64))
        st["dt"] = torch.tensor([st["dtv"]], device="cuda", dtype=F64)
        st["out"] = _views(plan, lev.state[1], 6)
        st["outg"] = _views(plan, st["g_new"], 3)
    else:
        plan, lev = _make(case, dense, keep_fluxes=1)
        fspec = WL.refine_boxes(spec, _refined(case, spec))
        fplan = H.Plan(fspec, stream=plan.torch_stream, keep_fluxes=1, coarse_fine=1,
                       **_params(case))
        fplan.layout_cache = {c: fplan.layout(c) for c in (3, 6)}
        amr = H.Amr(plan, fplan)
        flev = H.Level(fplan.empty_field(6), fplan.empty_field(6), fplan.empty_field(3))
        plan.fill(lev.state[0], 6)
        amr.interp(lev.state[0], flev.state[0], 6, "all")
        amr.interp(lev.grav, flev.grav, 3, "all")
        # fine data off its interpolant, so that both levels have their own
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 101)
        fac = 1.0 + 0.05 * torch.randn(_fine_extent(case), generator=gen, device="cuda", dtype=F64)
        for v in _views(fplan, flev.state[0], 6):
            v.mul_(fac.unsqueeze(1))
        st.update(plan=plan, lev=lev, fplan=fplan, flev=flev, amr=amr,
                  dt=torch.tensor([0.4 * _cfl(case, parts, dense, a[0])], device="cuda", dtype=F64),
                  dtn=torch.zeros(1, device="cuda", dtype=F64),
                  out=_views(plan, lev.state[1], 6) + _views(fplan, flev.state[1], 6))
    return st


def _fine_extent(case):
    return (case["nfine"],) + (2 * case["box"],) * 3


def run(st):
    kind, plan, lev, a = st["kind"], st["plan"], st["lev"], st["a"]
    lev.cur = 0
    if kind == "step":
        plan.advance(lev, a[:1], a[1:2], st["dt"], None, st["dtn"])
        return st["out"] + [st["dtn"]]
    if kind == "run":
        lev.state[0].copy_(st["snap"])
        plan.run(lev, a, st["dt"], st["steps"])
        return st["out"] + [st["dt"]]
    if kind == "host":
        dtn = plan.step_host_valid(lev, st["h_in"], st["h_out"], st["av"][0], st["av"][1], st["dt"])
        return [st["h_out"], dtn]
    if kind == "poisson":
        st["ps"].solve(lev.state[0], st["case"].get("a", A0), st["g"], warm_start=False)
        return st["out"]
    if kind == "cosmo":
        # Steps 2 to 6 of the single-level algorithm with g^n in hand
        ps, x, u, dt = st["ps"], st["x"], st["u"], st["dtv"]
        a0, a1 = st["av"]
        ah = 0.5 * (a0 + a1)
        x.copy_(st["x0"])
        u.copy_(st["u0"])
        plan.predict(lev, a[:1], a[1:2], st["dt"], lev.grav)
        ps.pm_kick_drift(x, u, st["gd0"], a0, ah, dt)
        ps.pm_deposit(x, st["m"], st["rho"])
        ps.solve(lev.state[1], a1, st["g_new"], warm_start=False, rho_dm=st["rho"],
                 g_dense=st["gd"])
        ps.pm_kick_estdt(x, u, st["gd"], ah, a1, dt, st["pdt"])
        plan.correct(lev, a[:1], a[1:2], st["dt"], lev.grav, st["g_new"], st["dtn"])
        return st["out"] + st["outg"] + [x, u, st["rho"], st["pdt"], st["dtn"]]
    st["flev"].cur = 0
    st["amr"].step(lev, st["flev"], a[:1], a[1:2], st["dt"], st["dtn"])
    return st["out"] + [st["dtn"]]


# ---------------------------------------------------------------- work and tolerance
def work(case):
    spec, _ = _parts(case)
    cells = spec.valid_cells()
    kind, prec = case["kind"], case["precision"]
    if kind in ("step", "run", "host"):
        n = case.get("steps", 1)
        by = (96 if case["level"] == "sod" else 120) * cells * n
        return {"bytes": by, "flops": FLOPS[prec] * cells * n}
    # a solve to 1e-12 takes about 12 cycles of 4 sweeps (9 operations a cell),
    # a residual, a restriction and a prolongation, over grids that sum to 8/7
    solve = 12 * 60 * 8 / 7
    if kind == "poisson":
        return {"bytes": (8 + 24) * cells, "flops": solve * cells}
    if kind == "cosmo":
        # gas 6 in, 6 out, g^n and g^{n+1}; particles 7 in, 6 out; dense g and rho
        return {"bytes": (96 + 48 + 104 + 8 + 32) * cells,
                "flops": (FLOPS[prec] + 44 + 250 + solve) * cells}
    fine = case["nfine"] * (2 * case["box"]) ** 3
    return {"bytes": 120 * (cells + fine), "flops": FLOPS[prec] * (cells + fine)}


def tolerance(case):
    """Measured against exact(): FP64 states agree to 1e-16 in the 2-norm, and
    another order of operations may move a limiter or sampling branch of a
    single cell (1e-12, the repository's own bar); mixed ones to 0.4e-7 to
    1.5e-7, single cells at strong jumps to 1e-3 where a branch differs.  The
    solve stops at a relative residual of 1e-12: 2e-13 to 4e-13 in g."""
    if case["kind"] == "poisson":
        return {"rel": 4e-12, "max": 1e-10}
    if case["precision"] == "fp64":
        return {"rel": 1e-12, "max": 1e-9}
    return {"rel": 6e-7, "max": 2e-3}


# ---------------------------------------------------------------- the scheme in FP64 torch
# Dense arrays (..., z, y, x); a shift wraps around, so that periodic domains
# need no ghost cells and other arrays carry four ghost layers of their own.
DIM = (2, 1, 0)      # axis of x, y, z in a (z, y, x) array


def _sh(q, d, o):
    """Value of the cell o further along direction d."""
    return torch.roll(q, -o, q.dim() - 3 + DIM[d])


class _K:
    def __init__(self, case):
        self.gamma = 1.4 if case["level"] == "sod" else 5.0 / 3.0
        self.gm1 = self.gamma - 1.0
        self.k = (self.gamma + 1.0) / (2.0 * self.gamma)
        self.sd, self.sp, self.eta, self.cfl = 1e-10, 1e-12, 1e-4, 0.5
        self.plm, self.linear = bool(case.get("plm")), bool(case.get("linear"))
        self.flat, self.genergy = bool(case.get("flat")), bool(case.get("genergy"))


def _cfl_state(K, S, a, dx):
    rho = S[0]
    p = torch.clamp(K.gm1 * S[5], min=K.sp)
    c = torch.sqrt(K.gamma * p / rho)
    return K.cfl * min(float((a * dx / ((S[1 + d] / rho).abs() + c)).min()) for d in range(3))


def _cfl(case, parts, dense, a):
    K = _K(case)
    return min(_cfl_state(K, d[0], a, p[2]) for p, d in zip(parts, dense))


def _prims(K, S):
    rho = S[0]
    return torch.stack([rho, S[1] / rho, S[2] / rho, S[3] / rho,
                        torch.clamp(K.gm1 * S[5], min=K.sp)])


def _mc(sm, s0, sp):
    dc, dl, dr = 0.5 * (sp - sm), s0 - sm, sp - s0
    m = torch.minimum(dc.abs(), 2 * torch.minimum(dl.abs(), dr.abs()))
    return torch.where(dl * dr > 0, torch.copysign(m, dc), torch.zeros_like(m))


def _profile(K, q, d):
    """Edge values and curvature of every cell's profile along d."""
    s1, s3 = _sh(q, d, -1), _sh(q, d, 1)
    d0 = _mc(s1, q, s3)
    if K.plm:
        return q - 0.5 * d0, q + 0.5 * d0, torch.zeros_like(q)
    edge = 0.5 * (s1 + q) - (d0 - _sh(d0, d, -1)) / 6
    sL, sR = edge, _sh(edge, d, 1)
    ext = (sR - q) * (q - sL) <= 0
    D, M = sR - sL, q - 0.5 * (sL + sR)
    lo = (~ext) & (D * M > D * D / 6)
    hi = (~ext) & ~lo & (-(D * D / 6) > D * M)
    nL = torch.where(ext, q, torch.where(lo, 3 * q - 2 * sR, sL))
    nR = torch.where(ext, q, torch.where(hi, 3 * q - 2 * sL, sR))
    return nL, nR, 6 * (q - 0.5 * (nL + nR))


def _chi(K, p, u, d, o):
    """Shock steepness of the cell o further along d."""
    P = [_sh(p, d, o + s) for s in (-2, -1, 1, 2)]
    um, up = _sh(u, d, o - 1), _sh(u, d, o + 1)
    dp = (P[2] - P[1]).abs()
    z = dp / torch.clamp((P[3] - P[0]).abs(), min=K.sp)
    w = torch.clamp(10 * (z - 0.75), 0.0, 1.0)
    on = (dp > 0.33 * torch.minimum(P[1], P[2])) & (um - up > 0)
    return torch.where(on, w, torch.zeros_like(w))


def _flat(K, q):
    f = None
    for d in range(3):
        p, u = q[4], q[1 + d]
        side = torch.where(_sh(p, d, 1) > _sh(p, d, -1), _chi(K, p, u, d, -1), _chi(K, p, u, d, 1))
        m = torch.maximum(_chi(K, p, u, d, 0), side)
        f = m if f is None else torch.maximum(f, m)
    return 1.0 - f


def _trace(K, q, g, d, dtdx, hdtp, src_u, src_p, fl):
    sL, sR, s6 = _profile(K, q, d)
    if fl is not None:
        sL, sR, s6 = fl * sL + (1 - fl) * q, fl * sR + (1 - fl) * q, fl * s6
    rho, un, pr = q[0], q[1 + d], q[4]
    c = torch.sqrt(K.gamma * pr / rho)
    lam = (un - c, un, un + c)
    sig = [x.abs() * dtdx for x in lam]
    c2 = c * c

    def ip(v, w):
        return sR[v] - 0.5 * sig[w] * ((sR[v] - sL[v]) - (1 - 2.0 / 3.0 * sig[w]) * s6[v])

    def im(v, w):
        return sL[v] + 0.5 * sig[w] * ((sR[v] - sL[v]) + (1 - 2.0 / 3.0 * sig[w]) * s6[v])

    n = 1 + d
    out = []
    for side in (1, 0):
        avg, edge, first, last = (ip, sR, 2, 0) if side else (im, sL, 0, 2)
        toward = [(x > 0) if side else (x < 0) for x in lam]
        ref = [torch.where(toward[first], avg(v, first), edge[v]) for v in range(5)]

        def gap(v, w):
            return torch.where(toward[w], ref[v] - avg(v, w), torch.zeros_like(rho))

        sgn = -1.0 if side else 1.0
        beta = (gap(4, last) + sgn * rho * c * gap(n, last)) * (0.5 / c2)
        b0 = gap(0, 1) - gap(4, 1) / c2
        r = [ref[0] - beta - b0, ref[1], ref[2], ref[3], ref[4] - c2 * beta]
        for t in (1, 2, 3):
            r[t] = (ref[t] - sgn * (c / rho) * beta) if t == n else ref[t] - gap(t, 1)
        for t in range(3):
            r[1 + t] = r[1 + t] - src_u * q[1 + t] + (hdtp * g[t] if g is not None else 0.0)
        r[4] = torch.clamp(r[4] - src_p * pr, min=K.sp)
        r[0] = torch.clamp(r[0], min=K.sd)
        out.append(torch.stack(r))
    return out[1], out[0]          # low face, high face


def _riemann(K, qL, qR, d):
    """Fluxes (rho, m_x, m_y, m_z, rhoE, rhoe, u, p) of the two-shock (or
    linearised) solution at x/t = 0."""
    rL, rR, uL, uR, pL, pR = qL[0], qR[0], qL[1 + d], qR[1 + d], qL[4], qR[4]
    cL, cR = torch.sqrt(K.gamma * pL / rL), torch.sqrt(K.gamma * pR / rR)
    CL, CR = rL * cL, rR * cR
    p = torch.clamp((CR * pL + CL * pR + CL * CR * (uL - uR)) / (CL + CR), min=K.sp)

    def W(C, ps, p):
        return C if K.linear else C * torch.sqrt(torch.clamp(1 + K.k * (p - ps) / ps, min=1e-10))

    for _ in range(0 if K.linear else 12):
        WL, WR = W(CL, pL, p), W(CR, pR, p)
        f = (uR + (p - pR) / WR) - (uL - (p - pL) / WL)
        ZL, ZR = 2 * WL**3 / (WL * WL + CL * CL), 2 * WR**3 / (WR * WR + CR * CR)
        p = torch.clamp(p - ZL * ZR * f / (ZL + ZR), min=K.sp)
    WL, WR = W(CL, pL, p), W(CR, pR, p)
    us = (pL - pR + WL * uL + WR * uR) / (WL + WR)

    def side(q, C, Wk, c, s):
        ro, uo, po = q[0], q[1 + d], q[4]
        if K.linear:
            rs = ro + (p - po) / (c * c)
        else:
            rs = 1 / (1 / ro - (p - po) / (Wk * Wk))
        rs = torch.clamp(rs, min=K.sd)
        cs = torch.sqrt(K.gamma * p / rs)
        shock = p > po
        S, Hd, T = uo - s * Wk / ro, uo - s * c, us - s * cs
        star = torch.where(shock, s * S < 0, (s * Hd < 0) & (s * T < 0))
        fan = ~shock & (s * Hd < 0) & ~(s * T < 0)
        w = torch.where(fan, Hd / (Hd - T), torch.zeros_like(Hd))
        w = torch.where(star, torch.ones_like(w), w)
        return [(1 - w) * x + w * y for x, y in ((ro, rs), (uo, us), (po, p))]

    gl, gr = side(qL, CL, WL, cL, 1.0), side(qR, CR, WR, cR, -1.0)
    up = us > 0
    mid = us == 0
    rg, ug, pg = (torch.where(mid, 0.5 * (x + y), torch.where(up, x, y)) for x, y in zip(gl, gr))
    rg, pg = torch.clamp(rg, min=K.sd), torch.clamp(pg, min=K.sp)
    vel = [torch.where(mid, 0.5 * (qL[1 + t] + qR[1 + t]), torch.where(up, qL[1 + t], qR[1 + t]))
           for t in range(3)]
    vel[d] = ug
    fr = rg * ug
    re = pg / K.gm1
    ke = 0.5 * rg * (vel[0]**2 + vel[1]**2 + vel[2]**2)
    F = [fr] + [fr * v for v in vel] + [ug * (re + ke + pg), ug * re, ug, pg]
    F[1 + d] = F[1 + d] + pg
    return torch.stack(F)


def _couple(K, q, terms):
    """Edge state q corrected by flux differences across its cell: terms of
    (coefficient, face fluxes along t, t)."""
    rn, m, en = q[0], [q[0] * q[1 + t] for t in range(3)], q[4] / K.gm1
    for c, F, t in terms:
        Fp = _sh(F, t, 1)
        rn = rn - c * (Fp[0] - F[0])
        m = [m[i] - c * (Fp[1 + i] - F[1 + i]) for i in range(3)]
        en = en - c * ((Fp[5] - F[5]) + 0.5 * (Fp[7] + F[7]) * (Fp[6] - F[6]))
    ok = rn >= K.sd
    new = [rn] + [x / rn for x in m] + [torch.clamp(K.gm1 * en, min=K.sp)]
    return torch.stack([torch.where(ok, x, y) for x, y in zip(new, q)])


def _fluxes(K, S, g, dx, a0, a1, dt):
    q = _prims(K, S)
    ah = 0.5 * (a0 + a1)
    dtp, adot = dt / ah, (a1 - a0) / ah
    fl = _flat(K, q) if K.flat else None
    lo, hi = [], []
    for d in range(3):
        m, p = _trace(K, q, g, d, dtp / dx, 0.5 * dtp, 0.5 * adot, 1.5 * K.gm1 * adot, fl)
        lo.append(m)
        hi.append(p)

    def solve(qm, qp, d):
        return _riemann(K, _sh(qp, d, -1), qm, d)

    Fn = [solve(lo[d], hi[d], d) for d in range(3)]
    third, half = dtp / (3 * dx), 0.5 * dtp / dx
    F2 = {}
    for d in range(3):
        for t in range(3):
            if t != d:
                m = _couple(K, lo[d], [(third, Fn[t], t)])
                p = _couple(K, hi[d], [(third, Fn[t], t)])
                F2[d, t] = solve(m, p, d)
    out = []
    for d in range(3):
        t1, t2 = [t for t in range(3) if t != d]
        terms = [(half, F2[t1, t2], t1), (half, F2[t2, t1], t2)]
        out.append(solve(_couple(K, lo[d], terms), _couple(K, hi[d], terms), d))
    return out


def _advance(K, S, g, dx, a0, a1, dt, full=True, g_new=None, fluxes=None):
    """One step on an array whose shifts stay inside it; the new state."""
    F = _fluxes(K, S, g, dx, a0, a1, dt) if fluxes is None else fluxes
    ah = 0.5 * (a0 + a1)
    div = sum((_sh(F[d][:6], d, 1) - F[d][:6]) / dx for d in range(3))
    pdv = sum(0.5 * (_sh(F[d][7], d, 1) + F[d][7]) * (_sh(F[d][6], d, 1) - F[d][6]) / dx
              for d in range(3))
    rho, m, rE, re = S[0], S[1:4], S[4], S[5]
    z = torch.zeros_like(m)
    G = g if g is not None else z
    kap = 2 - 3 * K.gm1
    expn = ah * (a1 - a0) * kap
    rs = rho - dt / ah * div[0]
    ms = (a0 * m - dt * div[1:4] + dt * rho * G) / a1
    mg = (m * G).sum(0)
    base = (a0 * a0 * rE - ah * dt * div[4] + expn * re)
    if K.genergy:
        mh = (a0 * m - dt * div[1:4]) / a1
        Es = base / a1**2 + 0.5 * ((ms * ms).sum(0) - (mh * mh).sum(0)) / rs
    else:
        Es = (base + dt * a0 * mg) / a1**2
    es = (a0 * a0 * re - ah * dt * (div[5] + pdv) + expn * re) / a1**2
    if not full:
        return torch.cat([rs[None], ms, Es[None], es[None]])
    return _finish(K, S, g, torch.cat([rs[None], ms, Es[None], es[None]]), g, a0, a1, dt)


def _finish(K, S, g0, P, g1, a0, a1, dt):
    """Gravity corrector and dual-energy synchronisation of a predictor P."""
    z = torch.zeros_like(S[1:4])
    go, gn = (g0 if g0 is not None else z), (g1 if g1 is not None else z)
    rs, ms, En, en = P[0], P[1:4], P[4], P[5]
    mn = ms + 0.5 * dt * (rs * gn - S[0] * go) / a1
    if K.genergy:
        En = En + 0.5 * ((mn * mn).sum(0) - (ms * ms).sum(0)) / rs
    else:
        En = En + 0.5 * dt * (a1 * (ms * gn).sum(0) - a0 * (S[1:4] * go).sum(0)) / a1**2
    ke = 0.5 * (mn * mn).sum(0) / rs
    big = En - ke > K.eta * En
    e2 = torch.where(big, En - ke, en)
    E2 = torch.where(big, En, en + ke)
    floor = K.sp / K.gm1
    low = e2 < floor
    e2 = torch.where(low, torch.full_like(e2, floor), e2)
    E2 = torch.where(low, e2 + ke, E2)
    return torch.cat([rs[None], mn, E2[None], e2[None]])


def _wrap(q, lo, hi):
    """Planes lo..hi of a periodic array."""
    return q.index_select(1, torch.arange(lo, hi, device=q.device) % q.shape[1])


def _slabs(K, S, g, dx, a0, a1, dt, **kw):
    """_advance over a periodic domain in slabs of planes (bounds the memory)."""
    nz = S.shape[1]
    step = max(8, int(4e6 / (S.shape[2] * S.shape[3])))
    if step >= nz:
        return _advance(K, S, g, dx, a0, a1, dt, **kw)
    out = []
    for z in range(0, nz, step):
        e = min(nz, z + step)
        gs = _wrap(g, z - 4, e + 4) if g is not None else None
        out.append(_advance(K, _wrap(S, z - 4, e + 4), gs, dx, a0, a1, dt, **kw)[:, 4:-4])
    return torch.cat(out, 1)


def _step_part(K, part, S, g, a0, a1, dt):
    if part[3] == "sod":           # outflow along x: four copies of the end cells
        pad = torch.cat([S[..., :1].expand(*S.shape[:-1], 4), S,
                         S[..., -1:].expand(*S.shape[:-1], 4)], -1)
        return _advance(K, pad, None, part[2], a0, a1, dt)[..., 4:-4]
    return _slabs(K, S, g, part[2], a0, a1, dt)


def _poisson_g(rho, dx, a):
    """-grad phi (centred) of the 7-point periodic Poisson equation."""
    n = rho.shape
    f = torch.fft.rfftn((rho - rho.mean()) / a)
    s = [torch.sin(math.pi * torch.fft.fftfreq(k, device=rho.device, dtype=F64))**2 for k in n]
    s[2] = torch.sin(math.pi * torch.arange(n[2] // 2 + 1, device=rho.device, dtype=F64) / n[2])**2
    lam = -(4 / dx**2) * (s[0].view(-1, 1, 1) + s[1].view(1, -1, 1) + s[2].view(1, 1, -1))
    lam[0, 0, 0] = 1.0
    f = f / lam
    f[0, 0, 0] = 0
    phi = torch.fft.irfftn(f, s=n)
    return torch.stack([-(_sh(phi, d, 1) - _sh(phi, d, -1)) * (0.5 / dx) for d in range(3)])


def _cic(x, n, dx):
    """(cell index, weight) of the 8 cells of every particle."""
    s = x / dx - 0.5
    i0 = torch.floor(s)
    w = (1 - (s - i0), s - i0)
    i = (torch.remainder(i0, n).long(), torch.remainder(i0 + 1, n).long())
    for o in range(8):
        b = (o & 1, (o >> 1) & 1, o >> 2)
        yield ((i[b[2]][2] * n + i[b[1]][1]) * n + i[b[0]][0],
               w[b[0]][0] * w[b[1]][1] * w[b[2]][2])


def _g_at(g, x, n, dx):
    out = torch.zeros_like(x)
    for idx, w in _cic(x, n, dx):
        out = out + w * g.reshape(3, -1)[:, idx]
    return out


def exact(case, seed):
    K = _K(case)
    spec, parts = _parts(case)
    dense = _dense(case, seed)
    kind, steps = case["kind"], case.get("steps", 1)
    a = _a(case, steps)
    if kind in ("step", "run", "host"):
        S = [d[0] for d in dense]
        dts = [_cfl(case, parts, dense, a[0])]
        for s in range(steps):
            S = [_step_part(K, p, q, d[1], a[s], a[s + 1], dts[s])
                 for p, q, d in zip(parts, S, dense)]
            dts.append(min(_cfl_state(K, q, a[s + 1], p[2]) for p, q in zip(parts, S)))
        out = _cut(spec, parts, S)
        if kind == "host":
            return [torch.cat([v.reshape(-1) for v in out]), dts[1]]
        return out + [torch.tensor(dts if kind == "run" else dts[1:], dtype=F64)]
    S0, g0 = dense[0]
    n, dx = case["n"], 1.0 / case["n"]
    if kind == "poisson":
        return _cut(spec, parts, [_poisson_g(S0[0], dx, A0)])
    if kind == "cosmo":
        dt = _cfl(case, parts, dense, a[0])
        ah = 0.5 * (a[0] + a[1])
        x, u, m = _particles(n, torch.Generator(device="cuda").manual_seed(int(seed) + 7919))
        P = _slabs(K, S0, g0, dx, a[0], a[1], dt, full=False)
        u = (a[0] * u + 0.5 * dt * _g_at(g0, x, n, dx)) / ah
        x = torch.remainder(x + dt / ah * u, 1.0)
        rho = torch.zeros(n**3, device="cuda", dtype=F64)
        for idx, w in _cic(x, n, dx):
            rho.index_add_(0, idx, m * w / dx**3)
        rho = rho.view(n, n, n)
        g1 = _poisson_g(P[0] + rho, dx, a[1])
        gp = _g_at(g1, x, n, dx)
        u = (ah * u + 0.5 * dt * gp) / a[1]
        pdt = min(0.5 * a[1] * dx / float(u.abs().max()), math.sqrt(dx / float(gp.abs().max())))
        new = _finish(K, S0, g0, P, g1, a[0], a[1], dt)
        return (_cut(spec, parts, [new]) + _cut(spec, parts, [g1])
                + [x, u, rho, torch.tensor([pdt], dtype=F64),
                   torch.tensor([_cfl_state(K, new, a[1], dx)], dtype=F64)])
    return _exact_amr(case, seed, K, spec, parts, dense, a)


def _interp2(q):
    """Dense refinement by 2 of dense cell values (nc, z, y, x): limited
    linear profiles that leave no fine value outside the cell's neighbours."""
    s = [_mc(_sh(q, d, -1), q, _sh(q, d, 1)) for d in range(3)]
    nb = torch.stack([q] + [_sh(q, d, o) for d in range(3) for o in (-1, 1)])
    hi, lo = nb.amax(0), nb.amin(0)
    dev = 0.25 * (s[0].abs() + s[1].abs() + s[2].abs())
    safe = torch.where(dev > 0, dev, torch.ones_like(dev))
    al = torch.minimum((hi - q) / safe, (q - lo) / safe).clamp(max=1.0)
    al = torch.where(dev > 0, al, torch.ones_like(al))
    nc, nz, ny, nx = q.shape
    out = torch.empty((nc, 2 * nz, 2 * ny, 2 * nx), device=q.device, dtype=F64)
    for o in range(8):
        b = (o & 1, (o >> 1) & 1, o >> 2)
        out[:, b[2]::2, b[1]::2, b[0]::2] = q + al * sum(
            s[d] * (0.25 if b[d] else -0.25) for d in range(3))
    return out


def _exact_amr(case, seed, K, spec, parts, dense, a):
    S0, g0 = dense[0]
    n, box, dx = case["n"], case["box"], 1.0 / case["n"]
    dt = 0.4 * _cfl(case, parts, dense, a[0])
    ah = 0.5 * (a[0] + a[1])
    ref = _refined(case, spec)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 101)
    fac = 1.0 + 0.05 * torch.randn(_fine_extent(case), generator=gen, device="cuda", dtype=F64)
    Fc = _fluxes(K, S0, g0, dx, a[0], a[1], dt)
    new = _advance(K, S0, g0, dx, a[0], a[1], dt, fluxes=Fc)
    Sf, gf = _interp2(S0), _interp2(g0)
    corner = [2 * spec.lo[b] for b in ref]
    covered = torch.zeros((n, n, n), device="cuda", dtype=torch.bool)
    for k, c in enumerate(corner):
        sl = tuple(slice(int(c[d]), int(c[d]) + 2 * box) for d in (2, 1, 0))
        Sf[(slice(None),) + sl] *= fac[k]
        covered[tuple(slice(s.start // 2, s.stop // 2) for s in sl)] = True
    ix = [[torch.arange(int(c[d]) - 4, int(c[d]) + 2 * box + 4, device="cuda") % (2 * n)
           for d in (2, 1, 0)] for c in corner]
    fine, coef = [], [dt / ah] + [dt / a[1]] * 3 + [ah * dt / a[1]**2] * 2
    coef = torch.tensor(coef, device="cuda", dtype=F64).view(6, 1, 1)
    for k, c in enumerate(corner):
        z, y, x = ix[k]
        cut = lambda q: q[:, z][:, :, y][:, :, :, x]  # noqa: E731
        Sb, gb = cut(Sf), cut(gf)
        Ff = _fluxes(K, Sb, gb, 0.5 * dx, a[0], a[1], dt)
        fine.append(_advance(K, Sb, gb, 0.5 * dx, a[0], a[1], dt, fluxes=Ff)[:, 4:-4, 4:-4, 4:-4])
        lo = c // 2
        for d in range(3):
            ax = 1 + DIM[d]
            for high in (0, 1):
                # the outside coarse cell, its face toward the fine box, and
                # the mean of the four fine fluxes through that face
                face = int(lo[d]) + (box if high else 0)
                cell = (face if high else face - 1) % n
                ff = Ff[d][:6].select(ax, 4 + (2 * box if high else 0))[:, 4:4 + 2 * box, 4:4 + 2 * box]
                avg = 0.25 * (ff[:, ::2, ::2] + ff[:, 1::2, ::2] + ff[:, ::2, 1::2] + ff[:, 1::2, 1::2])
                t = [e for e in (2, 1, 0) if e != d]
                sl = (slice(None),) + tuple(slice(int(lo[e]), int(lo[e]) + box) for e in t)
                fc = Fc[d][:6].select(ax, face % n)[sl]
                corr = coef * ((avg - fc) / dx) * (1.0 if high else -1.0)
                out = covered.select(DIM[d], cell)[sl[1:]]
                tgt = new.select(ax, cell)[sl]
                tgt += torch.where(out, torch.zeros_like(corr), corr)
    for k, c in enumerate(corner):
        f = fine[k]
        avg = sum(f[:, i::2, j::2, l::2] for i in (0, 1) for j in (0, 1) for l in (0, 1)) / 8
        lo = c // 2
        new[(slice(None),) + tuple(slice(int(lo[d]), int(lo[d]) + box) for d in (2, 1, 0))] = avg
    dtn = min([_cfl_state(K, new, a[1], dx)] + [_cfl_state(K, f, a[1], 0.5 * dx) for f in fine])
    return _cut(spec, parts, [new]) + [torch.stack(fine)] + [torch.tensor([dtn], dtype=F64)]
