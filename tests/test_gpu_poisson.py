"""GPU parity of the self-gravity solve (Sec. 3.4, nyx_poisson_*) against
the oracle: phi and g bitwise (same operations in the same order), the
V-cycle count, a warm start, and one step of the single-level algorithm
with self-gravity (Sec. 3.6: Step 1 solve, Step 2 predictor, Step 4 solve on
the predicted density, Step 6 corrector with the new g) in FP64."""
import numpy as np
import pytest

import oracle
from paper_1301_4498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
H = pytest.importorskip("paper_1301_4498_gb300.hydro")
torch = pytest.importorskip("torch")

FOUR_PI_G = 2.0


def _case():
    return W.tiled_box(n=64, box=32, sigma=1.0, seed=5, nsteps=2)


def test_solve_matches_the_oracle_bitwise():
    w = _case()
    a = 1 / 51
    phi_ref, g_ref, st = oracle.poisson_solve(w.level, oracle.PoissonParams(four_pi_G=FOUR_PI_G),
                                              w.state, a)
    oracle.fill_ghosts(w.level, g_ref)
    plan = H.Plan(w.level, gamma=w.gamma, cfl=w.cfl, precision="fp64")
    lev = H.make_level(plan, w.state, None)
    ps = H.Poisson(plan, four_pi_G=FOUR_PI_G)
    g = plan.empty_field(3)
    cyc, res = ps.solve(lev.current, a, g, warm_start=False)
    torch.cuda.synchronize()
    assert cyc == st["cycles"] and res <= 1e-12
    assert np.array_equal(ps.phi().cpu().numpy(), phi_ref)
    for x, y in zip(plan.from_device(g, 3), g_ref):
        assert np.array_equal(x, y)              # valid and ghost cells
    cyc2, _ = ps.solve(lev.current, a, g, warm_start=True)
    assert cyc2 == 0
    ps.close()
    plan.close()


def test_single_mode_on_the_gpu():
    n, k, amp = 32, (2, 1, 3), 0.1
    lev_spec = W.tiled_level(n, 16, dx=1.0 / n)
    z, y, x = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    theta = 2 * np.pi * (k[0] * x + k[1] * y + k[2] * z) / n
    rho = 1.0 + amp * np.sin(theta)
    states = []
    for b in range(lev_spec.nbox):
        arr = np.zeros(lev_spec.shape(b, 6))
        lo, hi = lev_spec.lo[b], lev_spec.hi[b]
        W.valid(arr)[0] = rho[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1]
        W.valid(arr)[5] = 1.0
        states.append(arr)
    plan = H.Plan(lev_spec, precision="fp64")
    lev = H.make_level(plan, states, None)
    ps = H.Poisson(plan, four_pi_G=1.0, tol=1e-13)
    g = plan.empty_field(3)
    ps.solve(lev.current, 1.0, g, warm_start=False)
    torch.cuda.synchronize()
    dx = 1.0 / n
    lam = -(4 / dx ** 2) * sum(np.sin(np.pi * kk / n) ** 2 for kk in k)
    phi = ps.phi().cpu().numpy()
    exact = amp * np.sin(theta) / lam
    assert np.abs((phi - phi.mean()) - exact).max() <= 1e-10 * np.abs(exact).max()
    ps.close()
    plan.close()


def test_self_gravity_step_matches_the_oracle():
    """Steps 1, 2, 4, 6 with the solve in the loop (FP64)."""
    w = _case()
    a0, a1 = float(w.a_sched[0]), float(w.a_sched[1])
    PP = oracle.PoissonParams(four_pi_G=FOUR_PI_G)
    P = oracle.OracleParams(gamma=w.gamma, cfl=w.cfl)
    phi, g0, _ = oracle.poisson_solve(w.level, PP, w.state, a0)
    oracle.fill_ghosts(w.level, g0)
    dt = oracle.estdt(w.level, P, w.state, a0)
    pred, _ = oracle.predict(w.level, P, w.state, g0, a_old=a0, a_new=a1, dt=dt)
    phi, g1, _ = oracle.poisson_solve(w.level, PP, pred, a1, phi)
    oracle.fill_ghosts(w.level, g1)
    ref, _ = oracle.correct(w.level, P, w.state, pred, g0, g1, a_old=a0, a_new=a1, dt=dt)

    plan = H.Plan(w.level, gamma=w.gamma, cfl=w.cfl, precision="fp64")
    lev = H.make_level(plan, w.state, None)
    ps = H.Poisson(plan, four_pi_G=FOUR_PI_G)
    gn, gp = plan.empty_field(3), plan.empty_field(3)
    a = torch.tensor([a0, a1], dtype=torch.float64, device="cuda")
    d = torch.zeros(2, dtype=torch.float64, device="cuda")
    ps.solve(lev.current, a0, gn, warm_start=False)
    plan.estdt(lev, a[:1], d[:1])
    plan.predict(lev, a[:1], a[1:], d[:1], gn)
    ps.solve(lev.state[1 - lev.cur], a1, gp, warm_start=True)
    plan.correct(lev, a[:1], a[1:], d[:1], gn, gp, dt_next=d[1:])
    torch.cuda.synchronize()
    assert plan.status() == (0, 0)
    got = plan.from_device(lev.current, 6)
    for c in range(6):
        num = max(np.abs(W.valid(x)[c] - W.valid(y)[c]).max() for x, y in zip(got, ref))
        den = max(np.abs(W.valid(y)[c]).max() for y in ref)
        assert num <= 1e-12 * den, c
    ps.close()
    plan.close()


def test_mixed_refinement_matches_the_oracle():
    """Iterative refinement (residual and update in fixed point, FP32 V-cycles)
    reaches the same stopping test as the oracle's FP64 multigrid, in about as
    many cycles.  Two solutions whose residuals are both below tol max|f|
    differ by L^-1 of at most 2 tol max|f|; with tol = 1e-12 on this 64^3
    grid that is far below the 1e-9 gates on phi and g written here."""
    w = _case()
    a = 1 / 51
    PP = oracle.PoissonParams(four_pi_G=FOUR_PI_G)
    phi_ref, g_ref, st = oracle.poisson_solve(w.level, PP, w.state, a)
    oracle.fill_ghosts(w.level, g_ref)
    plan = H.Plan(w.level, gamma=w.gamma, cfl=w.cfl, precision="fp64")
    lev = H.make_level(plan, w.state, None)
    ps = H.Poisson(plan, four_pi_G=FOUR_PI_G, precision="mixed")
    g = plan.empty_field(3)
    cyc, res = ps.solve(lev.current, a, g, warm_start=False)
    torch.cuda.synchronize()
    assert res <= 1e-12 and cyc <= st["cycles"] + 2
    phi = ps.phi().cpu().numpy()
    d = (phi - phi.mean()) - (phi_ref - phi_ref.mean())
    assert np.abs(d).max() <= 1e-9 * np.abs(phi_ref - phi_ref.mean()).max()
    gmax = max(np.abs(W.valid(y)).max() for y in g_ref)
    for x, y in zip(plan.from_device(g, 3), g_ref):
        assert np.abs(W.valid(x) - W.valid(y)).max() <= 1e-9 * gmax
    cyc2, _ = ps.solve(lev.current, a, g, warm_start=True)
    assert cyc2 == 0
    ps.close()
    plan.close()


def test_mixed_single_mode_closed_form():
    n, k, amp = 32, (2, 1, 3), 0.1
    lev_spec = W.tiled_level(n, 16, dx=1.0 / n)
    z, y, x = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    theta = 2 * np.pi * (k[0] * x + k[1] * y + k[2] * z) / n
    states = []
    for b in range(lev_spec.nbox):
        arr = np.zeros(lev_spec.shape(b, 6))
        lo, hi = lev_spec.lo[b], lev_spec.hi[b]
        W.valid(arr)[0] = (1.0 + amp * np.sin(theta))[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1,
                                                      lo[0]:hi[0] + 1]
        W.valid(arr)[5] = 1.0
        states.append(arr)
    plan = H.Plan(lev_spec, precision="fp64")
    lev = H.make_level(plan, states, None)
    ps = H.Poisson(plan, four_pi_G=1.0, tol=1e-13, precision="mixed")
    cyc, res = ps.solve(lev.current, 1.0, None, warm_start=False)
    torch.cuda.synchronize()
    assert res <= 1e-13
    dx = 1.0 / n
    lam = -(4 / dx ** 2) * sum(np.sin(np.pi * kk / n) ** 2 for kk in k)
    phi = ps.phi().cpu().numpy()
    exact = amp * np.sin(theta) / lam
    assert np.abs((phi - phi.mean()) - exact).max() <= 1e-10 * np.abs(exact).max()
    ps.close()
    plan.close()
