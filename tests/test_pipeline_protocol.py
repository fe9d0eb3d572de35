"""Host-side model of the task form's warp roles (nyx_fused2.cuh): column
warps that run the stages of two neighbouring planes in each interval,
update warps and loading warps, meeting on named barriers.

Per work item of planes [zb, ze):
  * loading warps: ring planes zb-3 .. zb+1 and plane zb-1's frame, arrive on
    LOADED; then for c = zb .. ze wait on CONSUMED, write ring plane c+2 and
    plane c's frame, arrive on LOADED;
  * column warps, c = zb-2 .. ze: interval A runs S3(c) (c >= zb-1) and, past
    a wait on LOADED, S1(c+1) (c < ze); stage barrier; arrive on CONSUMED when
    c+1 < ze; interval B runs S4(c) and S2(c+1), waits on FREE when
    c >= zb+2 before it stores the fluxes of plane c-1 and z face c, and
    arrives on READY when c >= zb+1; stage barrier;
  * update warps: for p = zb .. ze-1 wait on READY, update plane p, arrive on
    FREE when p+1 < ze;
  * all meet on the CTA barrier before the next item.
Every buffer carries the plane it holds; each stage checks what it reads and,
for the intervals, that no stage beside it writes the same slot.
"""
import random

import pytest

COL, UPD, LD = "C", "U", "L"
WEIGHT = {COL: 512, UPD: 128, LD: 128}
ALL = {COL, UPD, LD}


def column_ops(zb, ze):
    ops = []
    for c in range(zb - 2, ze + 1):
        if c < ze:
            ops.append(("sync", "LOADED", {COL, LD}))
        ops.append(("A", c))
        if c + 1 < ze:
            ops.append(("arrive", "CONSUMED", {COL, LD}))
        if c >= zb + 2:
            ops.append(("sync", "FREE", {COL, UPD}))
        ops.append(("B", c))
        if c >= zb + 1:
            ops.append(("arrive", "READY", {COL, UPD}))
    return ops + [("sync", "ALL", ALL)]


def load_ops(zb, ze):
    ops = [("prologue",), ("write", zb - 1), ("arrive", "LOADED", {COL, LD})]
    for c in range(zb, ze + 1):
        ops += [("sync", "CONSUMED", {COL, LD}), ("write", c), ("arrive", "LOADED", {COL, LD})]
    return ops + [("sync", "ALL", ALL)]


def update_ops(zb, ze):
    ops = []
    for p in range(zb, ze):
        ops += [("sync", "READY", {COL, UPD}), ("update", p)]
        if p + 1 < ze:
            ops.append(("arrive", "FREE", {COL, UPD}))
    return ops + [("sync", "ALL", ALL)]


class Buffers:
    """Shared memory of one CTA: what each slot holds, and the hand-over state."""

    def __init__(self):
        self.ring, self.frame = {}, None
        self.pair = {}            # x, y traced states: plane % 3 -> plane
        self.zlo, self.zhi = {}, {}   # right / left half of z face slot % 3 -> face
        self.fn, self.fz, self.p1 = None, {}, None
        self.fzxy = {}
        self.traced = set()
        self.xy, self.zf = None, {}   # fluxes handed over, not yet updated
        self.updated = set()

    def a(self, c, zb, ze):
        reads, writes = [], []
        if c >= zb - 1:                      # S3(c)
            assert self.fn == c and self.pair[c % 3] == c
            assert self.zlo[c % 3] == c and self.zhi[(c + 1) % 3] == c + 1
            if c >= zb + 1:
                assert self.pair[(c - 1) % 3] == c - 1
                assert self.fz[c & 1] == c and self.fz[(c - 1) & 1] == c - 1
                reads.append(("pair", (c - 1) % 3))
            reads += [("pair", c % 3), ("zlo", c % 3), ("zhi", (c + 1) % 3)]
        if c < ze:                           # S1(c+1)
            t = c + 1
            for k in range(t - 2, t + 3):
                assert self.ring.get(k % 5) == k, f"trace {t}: ring plane {k} missing"
            assert self.frame == t, f"trace {t}: frame holds {self.frame}"
            writes += [("pair", t % 3), ("zlo", t % 3), ("zhi", (t + 1) % 3)]
        assert not set(reads) & set(writes), "S1 overwrites what S3 reads beside it"
        if c >= zb - 1:
            self.p1 = c
            if c >= zb:
                self.fzxy[c & 1] = c
        if c < ze:
            self.pair[t % 3] = self.zlo[t % 3] = t
            self.zhi[(t + 1) % 3] = t + 1
            self.traced.add(t)

    def b(self, c, zb, ze):
        if c >= zb - 1:                      # S4(c)
            assert self.p1 == c
            assert self.zlo[c % 3] == c and self.zhi[(c + 1) % 3] == c + 1
            if c >= zb + 1:
                assert self.pair[(c - 1) % 3] == c - 1
                assert self.fzxy[c & 1] == c and self.fzxy[(c - 1) & 1] == c - 1
                assert self.xy is None, "x, y fluxes overwritten before their update"
                self.xy = c - 1
            if c >= zb:
                old = self.zf.get(c & 1)
                assert old is None or old in self.updated, f"z face {old} overwritten"
                self.zf[c & 1] = c
        if c < ze:                           # S2(c+1)
            t = c + 1
            assert self.pair[t % 3] == t and self.zlo[t % 3] == t
            self.fn = t
            if t >= zb:
                assert self.zhi[t % 3] == t
                self.fz[t & 1] = t

    def update(self, p, ze):
        assert self.xy == p and self.zf[p & 1] == p and self.zf[(p + 1) & 1] == p + 1
        self.xy = None
        self.updated.add(p)              # face p is not read again
        if p == ze - 1:
            self.updated.add(p + 1)

    def write(self, c, zb, ze):
        k = c + 2
        old = self.ring.get(k % 5)
        if old is not None:
            for t in range(max(zb - 1, old - 2), min(ze, old + 2) + 1):
                assert t in self.traced, f"ring plane {old} overwritten before trace {t}"
        self.ring[k % 5] = k
        assert self.frame is None or self.frame in self.traced, "frame overwritten"
        self.frame = c


def simulate(items, rng, make=(column_ops, update_ops, load_ops)):
    prog = {r: [(op, n) for n, (zb, ze) in enumerate(items) for op in f(zb, ze)]
            for r, f in zip((COL, UPD, LD), make)}
    pos = {r: 0 for r in prog}
    buf = [Buffers() for _ in items]
    bars, blocked = {}, {}
    while True:
        ready = [r for r in prog if r not in blocked and pos[r] < len(prog[r])]
        if not ready:
            assert not blocked, f"deadlock: {blocked}"
            return
        r = rng.choice(ready)
        op, n = prog[r][pos[r]]
        pos[r] += 1
        zb, ze = items[n]
        if op[0] in ("sync", "arrive"):
            b = bars.setdefault(op[1], [])
            b.append(r)
            want = sum(WEIGHT[x] for x in op[2])
            assert sum(WEIGHT[x] for x in b) <= want, f"{op[1]}: {b}"
            if op[0] == "sync":
                blocked[r] = op[1]
            if sum(WEIGHT[x] for x in b) == want:
                assert set(b) == op[2], f"{op[1]} phase by {b}"
                for x in list(blocked):
                    if blocked[x] == op[1]:
                        del blocked[x]
                bars[op[1]] = []
        elif op[0] == "prologue":
            for k in range(zb - 3, zb + 1):
                buf[n].ring[k % 5] = k
        elif op[0] == "write":
            buf[n].write(op[1], zb, ze)
        elif op[0] == "update":
            buf[n].update(op[1], ze)
        else:
            getattr(buf[n], op[0].lower())(op[1], zb, ze)


ITEMS = [[(0, 1)], [(0, 2)], [(0, 3)], [(0, 8)], [(0, 64)], [(0, 1), (1, 2), (2, 5), (7, 9)],
         [(0, 112), (112, 128), (0, 16)], [(5, 6), (6, 8), (0, 5), (3, 4), (40, 43)]]


@pytest.mark.parametrize("items", ITEMS)
def test_roles_never_deadlock_or_overwrite(items):
    for seed in range(100):
        simulate(items, random.Random(seed))


def _move(f, find, by):
    """The op list of f with the first op matching `find` moved by `by` places."""
    def g(zb, ze):
        ops = f(zb, ze)
        i = next(k for k, op in enumerate(ops) if find(op))
        ops.insert(i + by, ops.pop(i))
        return ops
    return g


@pytest.mark.parametrize("mistake", [
    # inputs written before the trace that still reads the old ones
    (column_ops, update_ops, _move(load_ops, lambda o: o == ("sync", "CONSUMED", {COL, LD}), 1)),
    # fluxes stored before the update released the buffers
    (_move(column_ops, lambda o: o[:2] == ("sync", "FREE"), 1), update_ops, load_ops),
    # an update that does not wait for its fluxes
    (column_ops, _move(update_ops, lambda o: o[:2] == ("sync", "READY"), 1), load_ops),
])
def test_planted_mistakes_are_caught(mistake):
    caught = 0
    for seed in range(100):
        try:
            simulate([(0, 8)], random.Random(seed), mistake)
        except (AssertionError, KeyError):
            caught += 1
    assert caught > 0
