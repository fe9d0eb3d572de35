"""What an earlier call leaves in a plan does not change a later one: tile
shapes changed between replays of a run's graph."""
import numpy as np
import pytest

from paper_1301_4498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
H = pytest.importorskip("paper_1301_4498_gb300.hydro")
torch = pytest.importorskip("torch")

A = (0.02, 0.0201, 0.0202)


def _scalars(dt=0.0):
    return (torch.tensor(A, dtype=torch.float64, device="cuda"),
            torch.tensor([dt, 0.0, 0.0], dtype=torch.float64, device="cuda"))


def _plan(w, **kw):
    return H.Plan(w.level, gamma=w.gamma, cfl=w.cfl, precision="mixed", **kw)


def _cache(monkeypatch, tmp_path, **picks):
    """A tuning cache that answers extent -> (shape, CTAs per SM)."""
    props = torch.cuda.get_device_properties(0)
    prefix = f"{props.name}|sm{props.multi_processor_count}|mixed|v0|"
    f = tmp_path / "tune.json"
    f.write_text("{\n" + ",\n".join(
        f' "{prefix}{e[1:]}": {{"shape": {s}, "ctas_per_sm": {c}, "ns_per_zone": 1}}'
        for e, (s, c) in picks.items()) + "\n}\n")
    monkeypatch.setenv("NYX_TUNE_CACHE", str(f))


class _Graphed:
    """A level replayed from the same buffers through a plan's graph cache."""

    def __init__(self, plan, w):
        self.plan, self.lev = plan, H.make_level(plan, w.state, w.grav)
        self.start = self.lev.state[0].clone()
        self.a, self.d = _scalars()

    def run(self):
        self.lev.state[0].copy_(self.start)
        self.lev.cur = 0
        self.plan.counters(reset=True)
        self.plan.run(self.lev, self.a, self.d, 1, compute_dt0=True, use_graph=True)
        torch.cuda.synchronize()
        assert self.plan.status()[0] == H.NYX_OK
        return (self.plan.counters(reset=True)["launches"],
                self.plan.from_device(self.lev.current, 6))


def test_graphs_follow_the_tile_shape(tmp_path, monkeypatch):
    # two parts (one launch each), then one shape, then another
    _cache(monkeypatch, tmp_path, x32x32x32=(3, 1), x64x64x64=(4, 2))
    w = W.large_level(n=64, box=32, nfine=2, nsteps=1)
    plan = _plan(w, autotune=1)
    g = _Graphed(plan, w)
    g.run()                          # tunes
    n_parts, _ = g.run()
    assert plan.tune_info()[2] == 2
    for shape in (0, 5, 0):
        plan.set_tile_shape(shape)
        ref = _plan(w)
        ref.set_tile_shape(shape)
        n, got = g.run()
        n_ref, want = _Graphed(ref, w).run()
        assert n == n_ref == n_parts - 1
        for x, y in zip(got, want):
            assert np.array_equal(W.valid(x), W.valid(y))
        ref.close()
    plan.close()


def test_two_level_graphs_follow_the_tile_shapes():
    import test_gpu_amr as TG
    import test_oracle_amr as TA
    w, fine = TA._hierarchy()

    def run(cp, amr, lc, lf, start):
        lc.state[0].copy_(start[0])
        lf.state[0].copy_(start[1])
        lc.cur = lf.cur = 0
        a, d = scal
        amr.run(lc, lf, a, d, 1, use_graph=True)
        torch.cuda.synchronize()
        assert cp.status()[0] == H.NYX_OK
        return cp.from_device(lc.current, 6)

    scal = _scalars()
    cp, fp, amr, lc, lf = TG._setup(w, fine, precision="mixed")
    start = (lc.state[0].clone(), lf.state[0].clone())
    run(cp, amr, lc, lf, start)
    cp.set_tile_shape(0)
    fp.set_tile_shape(2)
    got = run(cp, amr, lc, lf, start)
    cq, fq, amq, mc, mf = TG._setup(w, fine, precision="mixed")
    cq.set_tile_shape(0)
    fq.set_tile_shape(2)
    want = run(cq, amq, mc, mf, start)
    for x, y in zip(got, want):
        assert np.array_equal(W.valid(x), W.valid(y))
    for o in (amr, fp, cp, amq, fq, cq):
        o.close()
