"""What an earlier call leaves in a plan does not change a later one: box
groups made by a run and by a host step, tile shapes changed between replays
of a run's graph, a tile shape chosen while a stream is being captured."""
import ctypes as C

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


def _run(plan, w, **kw):
    """One step from the workload's state: (launches, new valid cells)."""
    lev = H.make_level(plan, w.state, w.grav)
    a, d = _scalars()
    plan.counters(reset=True)
    plan.run(lev, a, d, 1, compute_dt0=True, use_graph=False)
    torch.cuda.synchronize()
    assert plan.status()[0] == H.NYX_OK
    return plan.counters(reset=True)["launches"], [W.valid(x) for x in
                                                   plan.from_device(lev.current, 6)]


def _host(plan, w, dt):
    """One overlapped host step: (launches, new valid cells)."""
    lev = H.make_level(plan, w.state, w.grav)
    h_in = torch.from_numpy(plan.pack_valid(w.state)).pin_memory()
    h_out = torch.empty_like(h_in).pin_memory()
    plan.counters(reset=True)
    plan.step_host_valid(lev, h_in, h_out, A[0], A[1], dt)
    assert plan.status()[0] == H.NYX_OK
    return plan.counters(reset=True)["launches"], plan.unpack_valid(h_out.numpy())


# 27 boxes of 32^3 (1.4 waves: host steps overlap, runs do not) and 1000 boxes
# of 16^3 (13 waves: both do, by rules of their own)
@pytest.mark.parametrize("n,box", [(96, 32), (160, 16)])
def test_host_steps_and_runs_group_the_boxes_in_either_order(n, box):
    w = W.tiled_box(n=n, box=box, nsteps=1)
    dt = 1e-5
    p, q = _plan(w), _plan(w)
    host_first, s0 = _host(p, w, dt)
    run_after, s1 = _run(p, w)
    run_first, s2 = _run(q, w)
    host_after, s3 = _host(q, w, dt)
    assert host_after == host_first and run_after == run_first
    # a host step's group adds a gather and an advance launch to the run's
    assert host_first > run_first
    for x, y in zip(s0, s3):
        assert np.array_equal(x, y)
    for x, y in zip(s1, s2):
        assert np.array_equal(x, y)
    p.close()
    q.close()


def _cache(monkeypatch, tmp_path, **picks):
    """A tuning cache that answers extent -> (shape, CTAs per SM)."""
    props = torch.cuda.get_device_properties(0)
    prefix = f"{props.name}|sm{props.multi_processor_count}|mixed|v0|"
    f = tmp_path / "tune.json"
    f.write_text("{\n" + ",\n".join(
        f' "{prefix}{e[1:]}": {{"shape": {s}, "ctas_per_sm": {c}, "ns_per_zone": 1}}'
        for e, (s, c) in picks.items()) + "\n}\n")
    monkeypatch.setenv("NYX_TUNE_CACHE", str(f))


def test_a_run_groups_the_boxes_by_the_tuned_shape(tmp_path, monkeypatch):
    # 8 x 8 tiles at one CTA per SM: 26 waves, 6 groups; the shape before
    # tuning has 13 waves, 3 groups
    _cache(monkeypatch, tmp_path, x16x16x16=(4, 1))
    w = W.tiled_box(n=160, box=16, nsteps=1)
    p, q = _plan(w, autotune=1), _plan(w, autotune=1)
    _run(p, w)                       # tunes
    lev = H.make_level(q, w.state, w.grav)
    a, d = _scalars(1e-5)
    q.advance(lev, a[:1], a[1:2], d[:1])  # tunes too, without groups
    assert p.tune_info() == q.tune_info() and p.tune_info()[2] == 1
    n_p, s_p = _run(p, w)
    n_q, s_q = _run(q, w)
    assert n_p == n_q
    for x, y in zip(s_p, s_q):
        assert np.array_equal(x, y)
    p.close()
    q.close()


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


def test_a_tile_shape_chosen_while_a_stream_is_captured():
    # a blocking stream: work on the default stream would join the capture
    w = W.tiled_box(n=64, box=32, nsteps=1)
    s = C.c_void_p()
    assert int(torch.cuda.cudart().cudaStreamCreate(C.addressof(s))) == 0
    stream = torch.cuda.ExternalStream(s.value)
    plan = _plan(w, stream=stream)
    lev = H.make_level(plan, w.state, w.grav)
    a, d = _scalars(1e-5)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        plan.set_tile_shape(5)       # its work list is made and uploaded here
        plan.advance(lev, a[:1], a[1:2], d[:1])
    graph.replay()
    torch.cuda.synchronize()
    assert plan.status()[0] == H.NYX_OK
    ref = _plan(w)
    ref.set_tile_shape(5)
    rl = H.make_level(ref, w.state, w.grav)
    ref.advance(rl, a[:1], a[1:2], d[:1])
    for x, y in zip(plan.from_device(lev.current, 6), ref.from_device(rl.current, 6)):
        assert np.array_equal(W.valid(x), W.valid(y))
    del graph
    plan.close()
    ref.close()
    torch.cuda.cudart().cudaStreamDestroy(s.value)
