"""The splits of the work at the sizes where they can go wrong: columns cut
down to single planes, ghost rectangles and flattening columns cut into
pieces, scheme variants with their own instantiation, non-finite fluxes, and
the mixed Poisson solve on grids that its tiles do not divide, with other
sweep counts, from a given potential, at scales that fixed point cannot hold,
at tolerances near rounding, on a long domain, with a second solver alive and
without memory for its fused form."""
import itertools

import numpy as np
import pytest

import oracle
from gates import MIXED_GATES
from paper_1301_4498_gb300 import workloads as W

import test_oracle_amr as TA

pytestmark = pytest.mark.gpu
H = pytest.importorskip("paper_1301_4498_gb300.hydro")
torch = pytest.importorskip("torch")


def _boxes(extents, sigma=0.5, seed=11, bc=None):
    """Independent comoving boxes (or one box with boundary types bc)."""
    lev = (W.single_box_level(*extents[0], 1.0 / 64, bc) if bc
           else W.independent_boxes_level(extents, 1.0 / 64))
    S, G = [], []
    for b, (nx, ny, nz) in enumerate(extents):
        s, g = W._patch_state(lev, b, W.comoving_fields((nz, ny, nx), sigma, seed + b, 1.0 / 64))
        S.append(s)
        G.append(g)
    return lev, S, G


def _step(lev, S, G, dt, **kw):
    """One step of a given dt: the plan and the new state per box."""
    plan = H.Plan(lev, gamma=5.0 / 3.0, cfl=0.5, **kw)
    L = H.make_level(plan, S, G)
    a = torch.tensor([0.02, 0.0201], dtype=torch.float64, device="cuda")
    d = torch.tensor([dt, 0.0], dtype=torch.float64, device="cuda")
    plan.run(L, a, d, 1, compute_dt0=False, use_graph=False)
    torch.cuda.synchronize()
    return plan, plan.from_device(L.current, 6)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("extent", [(4, 4, 4), (8, 8, 6), (18, 10, 16), (34, 6, 30)])
def test_cut_columns_give_the_bits_of_whole_ones(extent, precision):
    # alone, the box's columns are cut until every SM has an item; among 1000
    # others they stay whole: the same cells from the same operations
    fill = [(16, 8, 4)] * 1000
    lev, S, G = _boxes([extent])
    p1, one = _step(lev, S, G, 1e-5, precision=precision)
    s0, g0 = S[0], G[0]
    lev2 = W.independent_boxes_level([extent] + fill, 1.0 / 64)
    f = W.comoving_fields((4, 8, 16), 0.5, 3, 1.0 / 64)
    s1, g1 = W._patch_state(lev2, 1, f)
    p2, many = _step(lev2, [s0] + [s1] * len(fill), [g0] + [g1] * len(fill), 1e-5,
                     precision=precision)
    assert p1.status() == (0, 0) and p2.status() == (0, 0)
    assert np.array_equal(W.valid(one[0]), W.valid(many[0]))
    p1.close()
    p2.close()


@pytest.mark.parametrize("bc", [(0,) * 6, (1,) * 6, (1, 0, 1, 1, 0, 1)])
@pytest.mark.parametrize("extent", [(4, 6, 8), (6, 130, 38), (130, 34, 6), (64, 64, 64)])
def test_cut_ghost_rectangles(extent, bc):
    lev, S, _ = _boxes([extent], bc=bc)
    plan = H.Plan(lev, gamma=1.4, cfl=0.5)
    for ncomp in (6, 3, 2):
        ref = [S[0][:ncomp].copy()]
        dev = plan.to_device(ref, ncomp)
        plan.fill(dev, ncomp)
        torch.cuda.synchronize()
        got = plan.from_device(dev, ncomp)
        oracle.fill_ghosts(lev, ref)
        assert np.array_equal(got[0], ref[0])
    plan.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("extent", [(4, 4, 4), (32, 14, 6), (34, 16, 10), (70, 36, 30)])
def test_cut_flattening_columns(extent, precision):
    lev, S, G = _boxes([extent], sigma=1.0)
    P = oracle.OracleParams(gamma=5.0 / 3.0, cfl=0.5, flattening=1)
    plan, got = _step(lev, S, G, 1e-5, precision=precision, flattening=True)
    assert plan.status() == (0, 0)
    ref = oracle.advance(lev, P, S, G, a_old=0.02, a_new=0.0201, dt=1e-5)[0]
    tol = 1e-12 if precision == "fp64" else MIXED_GATES["linf"]
    for c in range(6):
        g, r = W.valid(got[0])[c], W.valid(ref[0])[c]
        assert np.abs(g - r).max() <= tol * np.abs(r).max()
    plan.close()


@pytest.mark.parametrize("plm,linear,flat", list(itertools.product((0, 1), repeat=3)))
def test_variants_of_the_mixed_default_shape(plm, linear, flat):
    lev, S, G = _boxes([(18, 10, 14)], sigma=0.7)
    kw = dict(grav_energy=1, reconstruction=plm, riemann_solver=linear)
    P = oracle.OracleParams(gamma=5.0 / 3.0, cfl=0.5, flattening=flat, **kw)
    plan, got = _step(lev, S, G, 1e-5, precision="mixed", flattening=bool(flat), grav_energy=1,
                      reconstruction="plm" if plm else "ppm",
                      riemann_solver="linear" if linear else "two_shock")
    assert plan.status() == (0, 0) and plan.tile_shape()[0] == 3
    ref = oracle.advance(lev, P, S, G, a_old=0.02, a_new=0.0201, dt=1e-5)[0]
    for c in range(6):
        g, r = W.valid(got[0])[c], W.valid(ref[0])[c]
        assert np.abs(g - r).max() <= MIXED_GATES["linf"] * np.abs(r).max()
    plan.close()


@pytest.mark.parametrize("comp,value", [(0, np.nan), (1, np.nan), (1, np.inf), (2, -np.inf),
                                        (5, np.nan), (5, np.inf)])
@pytest.mark.parametrize("where", [(0, 0, 0), (17, 9, 13), (9, 7, 6)])
def test_non_finite_cells_reach_the_status(where, comp, value):
    lev, S, G = _boxes([(18, 10, 14)])
    i, j, k = where
    W.valid(S[0])[comp, k, j, i] = value
    plan, _ = _step(lev, S, G, 1e-5, precision="mixed")
    rc, flags = plan.status()
    assert rc != 0 and flags != 0
    plan.close()


def test_interpolation_ignores_nan_neighbours_as_the_oracle_does():
    w, fine = TA._hierarchy()
    cp = H.Plan(w.level, precision="fp64", keep_fluxes=1)
    fp = H.Plan(fine, stream=cp.torch_stream, precision="fp64", keep_fluxes=1, coarse_fine=1)
    amr = H.Amr(cp, fp)
    cs = TA._filled(w.level, w.state)
    rng = np.random.default_rng(4)
    for s in cs:
        for c in range(6):
            for z, y, x in rng.integers(0, s.shape[1], (40, 3)):
                s[c, z, y, x] = np.nan
    ref = oracle.amr_interp(w.level, cs, fine, TA._fine_empty(fine, 6), "all")
    dev = fp.empty_field(6)
    amr.interp(cp.to_device(cs, 6), dev, 6, "all")
    torch.cuda.synchronize()
    for g, r in zip(fp.from_device(dev, 6), ref):
        assert np.array_equal(g, r, equal_nan=True)
    amr.close(); fp.close(); cp.close()


def _spectral_phi(f, h):
    """Zero-mean solution of the 7-point Laplacian: the operator is diagonal in
    Fourier space."""
    F = np.fft.fftn(f)
    lam = 0.0
    for ax, n in enumerate(f.shape):
        s = [1, 1, 1]
        s[ax] = n
        lam = lam - (4.0 / h**2) * (np.sin(np.pi * np.arange(n) / n)**2).reshape(s)
    lam = np.broadcast_to(lam, f.shape).copy()
    lam[0, 0, 0] = 1.0
    F /= lam
    F[0, 0, 0] = 0.0
    return np.fft.ifftn(F).real


@pytest.mark.parametrize("n,prm,scale,warm", [
    (8, {}, 1.0, False), (20, {}, 1.0, False), (36, {}, 1.0, True), (64, {}, 1.0, False),
    (100, {}, 1.0, False), (128, {}, 1.0, True),
    (48, dict(pre=1, post=1), 1.0, False), (48, dict(pre=3, post=2), 1.0, True),
    (48, dict(pre=0, post=3), 1.0, False), (48, dict(pre=2, post=0), 1.0, True),
    (32, {}, 1e-14, False), (32, {}, 1e12, True), (32, {}, 1e-30, False), (32, {}, 1e25, True)])
def test_mixed_poisson_solve(n, prm, scale, warm):
    lev = W.single_box_level(n, n, n, 1.0 / n)
    rng = np.random.default_rng(n)
    arr = np.zeros(lev.shape(0, 6))
    W.valid(arr)[0] = np.exp(rng.standard_normal((n, n, n)))
    plan = H.Plan(lev, precision="fp64")
    L = H.make_level(plan, [arr], None)
    tol = 1e-11
    ps = H.Poisson(plan, four_pi_G=scale, precision="mixed", tol=tol, max_cycles=200, **prm)
    if warm:  # from the potential of another density
        other = np.zeros_like(arr)
        W.valid(other)[0] = 1.0 + rng.random((n, n, n))
        ps.solve(plan.to_device([other], 6), 0.5, None, warm_start=False)
    cyc, res = ps.solve(L.current, 0.5, None, warm_start=warm)
    phi = ps.phi().cpu().numpy()
    rho = W.valid(arr)[0]
    f = scale / 0.5 * (rho - rho.mean())
    ref = _spectral_phi(f, 1.0 / n)
    phi = phi - phi.mean()
    # a residual of max norm r leaves an error of at most 0.26 l^2 r (the zero-mean
    # inverse of the operator on a periodic box of side l = 1)
    assert 0 < cyc and res <= tol
    assert np.abs(phi - ref).max() <= 0.26 * tol * np.abs(f).max() + 1e-12 * np.abs(ref).max()
    ps.close()
    plan.close()


def _poisson_box(n, seed, **prm):
    """(plan, solver, device state, spectral potential of its density, max|f|)
    of one periodic box of n = (nx, ny, nz) cells of width 1 / max(n)."""
    h = 1.0 / max(n)
    lev = W.single_box_level(*n, h)
    arr = np.zeros(lev.shape(0, 6))
    rho = np.exp(np.random.default_rng(seed).standard_normal(n[::-1]))
    W.valid(arr)[0] = rho
    plan = H.Plan(lev, precision="fp64")
    f = rho - rho.mean()
    return (plan, H.Poisson(plan, **prm), plan.to_device([arr], 6), _spectral_phi(f, h),
            np.abs(f).max())


def _solve_and_check(box, tol, warm=False):
    _, ps, state, ref, fmax = box
    cyc, res = ps.solve(state, 1.0, None, warm_start=warm)
    phi = ps.phi().cpu().numpy()
    # the bound of test_mixed_poisson_solve, l = 1
    assert res <= tol
    assert (np.abs(phi - phi.mean() - ref).max()
            <= 0.26 * tol * fmax + 1e-12 * np.abs(ref).max())
    return cyc, res


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("first,second", [(128, 96), (96, 128), (40, 128)])
def test_live_solvers_keep_their_own_tails(first, second, precision):
    # the coarse grids run in one CTA whose shared memory differs by grid: a
    # solver made later, or destroyed, must not narrow what an earlier one may use
    a = _poisson_box((first,) * 3, 1, precision=precision, tol=1e-11)
    b = _poisson_box((second,) * 3, 2, precision=precision, tol=1e-11)
    for box in (a, b, a):
        _solve_and_check(box, 1e-11)
    b[1].close()
    _solve_and_check(a, 1e-11)
    a[1].close()
    a[0].close()
    b[0].close()


def test_mixed_poisson_at_tolerances_near_rounding():
    # an uncorrelated density: FP64 sums leave a residual of about 1e-16 max|f|
    box = _poisson_box((128,) * 3, 3, precision="mixed", tol=2e-15, max_cycles=30)
    _solve_and_check(box, 2e-15)
    # the same density again: solved already, and left as it is
    before = box[1].phi()
    assert _solve_and_check(box, 2e-15, warm=True)[0] == 0
    assert torch.equal(before, box[1].phi())
    box[1].close()
    box[0].close()


@pytest.mark.parametrize("warm", [False, True])
def test_mixed_poisson_on_a_long_domain(warm):
    # 2048 x 16 x 16 cells at the default tolerance, a density of period 32
    # cells (so that it converges as one period does): the potential is 64^2
    # times smaller than a domain of this length allows
    n, h, per = (2048, 16, 16), 1.0 / 2048, 32
    rng = np.random.default_rng(8)
    cell = [np.exp(rng.standard_normal((16, 16, per))) for _ in range(2)]
    lev = W.single_box_level(*n, h)
    plan = H.Plan(lev, precision="fp64")
    ps = H.Poisson(plan, precision="mixed")
    for c in cell[:1 + warm]:
        arr = np.zeros(lev.shape(0, 6))
        W.valid(arr)[0] = np.tile(c, (1, 1, n[0] // per))
        cyc, res = ps.solve(plan.to_device([arr], 6), 1.0, None, warm_start=warm)
        assert res <= 1e-12
    f = c - c.mean()
    ref = np.tile(_spectral_phi(f, h), (1, 1, n[0] // per))
    phi = ps.phi().cpu().numpy()
    # (of length 32 h each period)
    assert (np.abs(phi - phi.mean() - ref).max()
            <= 0.26 * (per * h)**2 * 1e-12 * np.abs(f).max() + 1e-12 * np.abs(ref).max())
    ps.close()
    plan.close()


def test_interpolation_and_average_down_of_more_components_than_a_grid_holds():
    # components run along grid y, of at most 65535 blocks: two fields in turn
    n = 70000
    cl = W.single_box_level(8, 8, 8, 1.0 / 8)
    fl = W.refined_level(cl, [(0, (2, 2, 2), (3, 3, 3))])
    cp = H.Plan(cl, precision="fp64", keep_fluxes=1)
    fp = H.Plan(fl, stream=cp.torch_stream, precision="fp64", keep_fluxes=1, coarse_fine=1)
    amr = H.Amr(cp, fp)
    c2 = cp.empty_field(2)
    c2.copy_(torch.rand(c2.shape, dtype=torch.float64, device="cuda"))
    f2, back = fp.empty_field(2), cp.empty_field(2)
    amr.interp(c2, f2, 2, "all")
    amr.average_down(f2, back, 2)
    cn = c2.repeat(n // 2)            # one box: components follow one another
    fn, bn = fp.empty_field(n), cp.empty_field(n)
    amr.interp(cn, fn, n, "all")
    amr.average_down(fn, bn, n)
    assert torch.equal(fn, f2.repeat(n // 2)) and torch.equal(bn, back.repeat(n // 2))
    amr.close(); fp.close(); cp.close()


def test_mixed_poisson_without_memory_for_the_fused_sweeps():
    # 512^3: 3.7 GB of grids, 1.7 GB more for the fused sweeps and fixed point
    n = 512
    lev = W.single_box_level(n, n, n, 1.0 / n)
    plan = H.Plan(lev, precision="fp64")
    state = plan.empty_field(6)
    state.copy_(torch.rand(state.shape, dtype=torch.float64, device="cuda"))

    def solve(ps):
        cyc, res = ps.solve(state, 1.0, None, warm_start=False)
        phi = ps.phi()
        ps.close()
        assert res <= 1e-11
        return cyc, phi - phi.mean()

    want = solve(H.Poisson(plan, precision="mixed", tol=1e-11))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = torch.empty(torch.cuda.mem_get_info()[0] - 4600 * 2**20, dtype=torch.uint8,
                       device="cuda")
    ps = H.Poisson(plan, precision="mixed", tol=1e-11)
    left = torch.cuda.mem_get_info()[0]
    del held
    torch.cuda.empty_cache()
    assert left > 0.6e9               # the fused form's arrays were given back
    got = solve(ps)
    assert abs(got[0] - want[0]) <= 1
    # both residuals are below 1e-11 max|f| (< 1e-11), l = 1
    assert (got[1] - want[1]).abs().max() <= 2 * 0.26e-11
    plan.close()
