"""Host: the schedules that whole tapes are walked by, replayed against the hazards they must keep.

The kernels read records and do what they say: nothing on the device checks that a state has been written, or is
still there.  Here every record is executed on tags instead of numbers -- "h of step 7, layer 1" -- phase by phase:
what a task reads must carry the tag it needs before the phase begins, and nothing that one task of a phase writes
may be read or written by another of the same phase.
"""
import random
import struct

import pytest

from paper_1606_03401_b200 import binding as B

NONE = 0xffff
FWD, READ, BWD, LOAD_H, LOAD_X, DHA, CARRY = 1, 2, 3, 4, 5, 6, 7
ZERO = ("zero",)


class Replay:
    def __init__(self, desc, plan, room=0):
        self.L, self.t = desc.layers, desc.t
        self.gru = bool(desc.flags & B.MEBPTT_FLAG_GRU)
        self.cr = 2 if desc.dtype == B.MEBPTT_BF16 else 1
        self.info, records, launches = B.mebptt_test_schedule(desc, plan, room)
        self.records, self.launches = [bytes(r) for r in records], launches.tolist()
        self.plan, self.S, self.parts = plan, self.info["chunk"], self.info["parts"]
        self.mem = {}                       # part of a block -> tag; stages and carries by name
        self.slots = {}                     # operand slots of the pods (16-byte units), empty at each launch
        self.forwards, self.next_b = {}, [self.t] * self.L
        for l in range(self.L):
            self._put(self._h(self.info["init"], l), ("h", 0, l))
            self._put(self._c(self.info["init"], l), ("c", 0, l))
            for par in (0, 1):
                self.mem["carry", par, l] = ZERO

    # ---- where things lie ----
    def _range(self, loc, block, n):
        lo = loc + block * self.parts
        assert 0 <= lo and lo + n * self.parts <= self.info["n_blocks"]
        return range(lo, lo + n * self.parts)

    def _h(self, loc, l):
        return self._range(loc, l * (1 + self.cr), 1)

    def _c(self, loc, l):
        return self._range(loc, l * (1 + self.cr) + 1, self.cr)

    def _g(self, loc, l):
        return self._range(loc, self.L * (1 + self.cr) + 4 * l, 4)

    def _in(self, loc):
        return loc + (self.L * (1 + self.cr) + 4 * self.L) * self.parts

    def _put(self, cells, tag):
        for i in cells:
            self.mem[i] = tag

    # ---- a phase: reads against the state before it, then the writes ----
    def _begin(self):
        self.reads, self.writes = [], []

    def _need(self, task, cells, tag, where=None):
        mem = self.mem if where is None else where
        for i in (cells if isinstance(cells, range) else [cells]):
            assert mem.get(i) == tag, (task, i, mem.get(i), tag)
            self.reads.append((task, where is not None, i))

    def _give(self, task, cells, tag, slot=False):
        for i in (cells if isinstance(cells, range) else [cells]):
            self.writes.append((task, slot, i, tag))

    def _end(self):
        owner = {}
        for task, slot, i, tag in self.writes:
            assert owner.setdefault((slot, i), task) is task, ("written twice", task, i)
        for task, slot, i in self.reads:
            # (a task's own result may take the place of its operand only in memory, where one thread does both)
            w = owner.get((slot, i))
            assert w is None or (w is task and not slot), ("read and written", task, w, i)
        for task, slot, i, tag in self.writes:
            (self.slots if slot else self.mem)[i] = tag

    def _forward(self, task, k, l, src, dst, gates, copy):
        self._need(task, self._h(src, l), ("h", k - 1, l))
        if not self.gru:
            self._need(task, self._c(src, l), ("c", k - 1, l))
            self._give(task, self._c(dst, l), ("c", k, l))
        self._give(task, self._h(dst, l), ("h", k, l))
        if gates:
            self._give(task, self._g(dst, l), ("g", k, l))
        if copy:
            self._give(task, self._h(self._in(dst), l), ("h", k - 1, l))
            if not self.gru:
                self._give(task, self._c(self._in(dst), l), ("c", k - 1, l))
        self.forwards[k, l] = self.forwards.get((k, l), 0) + 1

    def _backward(self, task, k, l, sidx, src, dst, last_of_chunk, first_of_chunk):
        assert self.next_b[l] == k and sidx == (k - 1) % self.S
        self.next_b[l] -= 1
        self._need(task, self._g(src, l), ("g", k, l))
        self._need(task, self._h(dst, l), ("h", k - 1, l))
        if not self.gru:
            self._need(task, self._c(src, l), ("c", k, l))
            self._need(task, self._c(dst, l), ("c", k - 1, l))
        self._give(task, ("dz", l, sidx), ("dz", k, l))
        self._give(task, ("hs", l, sidx), ("h", k - 1, l))
        assert last_of_chunk == (k == self.t or sidx == self.S - 1) and first_of_chunk == (sidx == 0)
        if last_of_chunk:
            self._need(task, self._h(src, l), ("h", k, l))
            self._give(task, ("hs", l, sidx + 1), ("h", k, l))
        if first_of_chunk:
            self._give(task, ("carry", k & 1, l), ("dz", k, l))

    def _carried(self, k, l):
        return ("dz", k + 1, l) if k < self.t else ZERO

    def _chunk_done(self, chunk):
        steps = min(self.S, self.t - chunk * self.S)
        for l in range(self.L):
            assert self.next_b[l] == chunk * self.S
            for s in range(steps):
                assert self.mem["dz", l, s] == ("dz", chunk * self.S + s + 1, l)
                assert self.mem["hs", l, s] == ("h", chunk * self.S + s, l)
            assert self.mem["hs", l, steps] == ("h", chunk * self.S + steps, l)
        for s in range(steps):
            assert self.mem["dy", s] == ("dy", chunk * self.S + s + 1)

    def run(self):
        todo = -(-self.t // self.S) - 1
        for first, n, phases, chunk in self.launches:
            assert n % 64 == 0 and n <= (self.room if hasattr(self, "room") else 1 << 30)
            seen = (self._pods if self.info["pods"] else self._teams)(self.records[first:first + n])
            assert seen == phases
            if chunk >= 0:
                assert chunk == todo
                todo -= 1
                self._chunk_done(chunk)
        assert todo == -1
        want = {}
        for op in self.plan.tape():
            if op["kind"] == 1:
                for l in range(self.L):
                    want[int(op["k"]), l] = want.get((int(op["k"]), l), 0) + 1
        assert self.forwards == want and self.next_b == [0] * self.L

    # ---- the walking kernel: phases end with a flag, no phase straddles a window of 64 records ----
    def _teams(self, records):
        i = phases = 0
        while i < len(records):
            if records[i][0] == 0:
                i = (i // 64 + 1) * 64
                continue
            start = i
            self._begin()
            while True:
                task = (i,) + struct.unpack("<BBBxiIIIII4x", records[i])
                self._team_task(task)
                i += 1
                if task[3] & 1:
                    break
            assert i - start <= 8 and start // 64 == (i - 1) // 64
            self._end()
            phases += 1
        return phases

    def _team_task(self, task):
        _, kind, l, flags, k, src, dst, sidx, _, _ = task
        if kind == FWD:
            if l:
                self._need(task, self._h(dst, l - 1), ("h", k, l - 1))
            self._forward(task, k, l, src, dst, flags & 2, flags & 4)
        elif kind == READ:
            self._need(task, self._h(src, l), ("h", k, self.L - 1))
            self._give(task, ("dy", sidx), ("dy", k))
        else:
            assert kind == BWD
            self._backward(task, k, l, sidx, src, dst, bool(flags & 8), bool(flags & 16))
            if flags & 8:
                self._need(task, ("carry", (k + 1) & 1, l), self._carried(k, l))
            else:
                self._need(task, ("dz", l, sidx + 1), ("dz", k + 1, l))
            if l + 1 < self.L:
                self._need(task, ("dz", l + 1, sidx), ("dz", k, l + 1))
            else:
                self._need(task, ("dy", sidx), ("dy", k))

    # ---- the pod kernel: a header, then its tasks; results go to slots of shared memory ----
    def _pods(self, records):
        self.slots = {}
        i = phases = 0
        while i < len(records):
            h = records[i]
            n, cells, sums, n_h, n_p, n_x, r, x, products = h[:9]
            main, load, carry, bwd = struct.unpack("<IIII", h[12:28])
            if n == 0:
                i = (i // 64 + 1) * 64
                continue
            assert i // 64 == (i + n) // 64
            tasks = [(i + 1 + j,) + struct.unpack("<BBBxiIIHHHHIHH", records[i + 1 + j]) for j in range(n)]
            self._begin()
            kinds, count = [], {"h": 0, "p": 0, "x": 0}
            index = {"main": 0, "load": 0, "carry": 0, "bwd": 0, "r": 0, "x": 0}
            for j, task in enumerate(tasks):
                kind, l = task[1], task[2]
                kinds.append(kind)
                nib = (j + 1) << (4 * l)
                if kind in (FWD, BWD):
                    assert not index["main"] >> (4 * l) & 15
                    index["main"] |= nib
                    index["bwd"] |= nib if kind == BWD else 0
                elif kind == LOAD_H:
                    assert not index["load"] >> (4 * l) & 15
                    index["load"] |= nib
                elif kind == CARRY:
                    index["carry"] |= nib
                elif kind in (READ, LOAD_X):
                    key = "r" if kind == READ else "x"
                    assert not index[key]
                    index[key] = j + 1
                self._pod_task(task, count)
            busy = [q for q in kinds if q in (FWD, READ, BWD, DHA, CARRY)]
            assert products == len(busy) and kinds[:products] == busy
            assert bool(cells) == any(q in (BWD, DHA, CARRY) for q in kinds) and bool(sums) == any(q in (FWD, READ) for q in kinds)
            assert (n_h, n_p, n_x) == (count["h"], count["p"], count["x"])
            assert (main, load, carry, bwd, r, x) == tuple(index[q] for q in ("main", "load", "carry", "bwd", "r", "x"))
            self._end()
            phases += 1
            i += n + 1
        return phases

    def _pod_task(self, task, count):
        _, kind, l, flags, k, src, dst, sidx, sa, sb, so, _, red, _ = task
        if kind == FWD:
            self._need(task, sa, ("x", k) if l == 0 else ("h", k, l - 1), self.slots)
            self._need(task, sb, ("h", k - 1, l), self.slots)
            self._forward(task, k, l, src, dst, flags & 1, flags & 2)
            if so != NONE:
                self._give(task, so, ("h", k, l), True)
                count["h"] += 1
        elif kind == READ:
            self._need(task, sb, ("h", k, self.L - 1), self.slots)
            self._give(task, so, ("dy", k), True)
            self._give(task, ("dy", sidx), ("dy", k))
        elif kind == DHA:
            self._need(task, sa, ("dy", k), self.slots)
            assert so == red
            self._give(task, so, ("above", k, self.L - 1), True)
            count["p"] += 1
        elif kind == CARRY:
            cell = ("carry", (k + 1) & 1, l) if sidx == NONE else ("dz", l, sidx)
            self._need(task, cell, ("dz", k + 1, l))
            self._give(task, so, ("own", k, l), True)
            count["p"] += 1
        elif kind == BWD:
            self._backward(task, k, l, sidx, src, dst, bool(flags & 8), bool(flags & 16))
            assert bool(flags & 4) == (k == self.t)
            if k < self.t:
                self._need(task, sa, ("own", k, l), self.slots)
            self._need(task, sb, ("above", k, l), self.slots)
            if l:
                self._give(task, red, ("above", k, l - 1), True)
                count["p"] += 1
            if not flags & 16:
                self._give(task, so, ("own", k - 1, l), True)
                count["p"] += 1
        elif kind == LOAD_H:
            tag = self.mem.get(self._h(src, l)[0])
            assert tag is not None and tag[0] == "h" and tag[2] == l
            self._need(task, self._h(src, l), tag)
            self._give(task, so, tag, True)
            count["h"] += 1
        elif kind == LOAD_X:
            self._give(task, so, ("x", k), True)
            count["x"] += 1
        else:
            assert kind == 0          # an empty phase


def _desc(rng, route):
    while True:
        dtype, gru = rng.choice(("fp32", "bf16")), rng.random() < 0.3
        hidden = rng.choice((24, 40, 64, 130, 200, 256)) if route == "pods" else rng.choice((300, 515, 301, 700))
        desc = B.make_desc(rng.choice((1, 1, 2, 2, 3, 4)), rng.choice((9, 40, 77)), hidden, rng.choice((5, 29)),
                           rng.choice((1, 3, 9, 20, 40)), rng.choice((1, 2, 5, 17, 33, 70, 130)), dtype,
                           flags=B.MEBPTT_FLAG_GRU if gru else 0)
        plan = _plan(rng, desc)
        if plan is not None and B.mebptt_test_route(desc, plan)["route"] == route:
            return desc, plan


def _plan(rng, desc):
    t = desc.t
    kind = rng.choice(("hsm", "ism", "msm", "msm3", "full", "chen", "exact", "exact", "whole"))
    if kind == "full":
        return B.mebptt_plan(t, t, B.MEBPTT_ISM)
    if kind == "chen":
        return B.mebptt_plan_chen_sqrt(t, 4, rng.choice((0, 3)))
    if kind == "exact":
        return B.mebptt_plan_bytes_exact(desc, rng.randint(3, 40) * B.mebptt_lstm_unit_bytes(desc), rng.random() < 0.5)
    if kind == "whole":
        plan = B.mebptt_plan(t, 8, B.MEBPTT_MSM)
        try:
            return B.mebptt_plan_for_bytes(desc, int(B.mebptt_lstm_workspace_bytes(desc, plan) * rng.uniform(0.5, 1.5)),
                                           B.MEBPTT_MSM, include_working=True)
        except B.MebpttError:
            return None
    m = rng.choice((1, 2, 4, 7, 15, 40)) if t < 100 else rng.choice((4, 7, 15, 40))
    return B.mebptt_plan_ex(t, m, B.MODES[kind[:3]], 4, 3 if kind == "msm3" else 0)


@pytest.mark.parametrize("route", ["pods", "teams"])
def test_schedules_keep_every_hazard(route):
    rng = random.Random(7)
    for _ in range(150):
        desc, plan = _desc(rng, route)
        room = rng.choice((0, 0, 256, 512))
        replay = Replay(desc, plan, room)
        replay.room = room or replay.info["room"]
        replay.run()


@pytest.mark.parametrize("route", ["pods", "teams"])
def test_the_replay_notices_a_mistake(route):
    """A forward task that reads its state one block off, or (teams) begins a phase too early."""
    rng = random.Random(3)
    ran = 0
    while ran < 20:
        desc, plan = _desc(rng, route)
        replay = Replay(desc, plan)
        headers = set()
        if route == "pods":
            for first, n, _, _ in replay.launches:
                i = first
                while i < first + n:
                    headers.add(i)
                    i = i + 1 + replay.records[i][0] if replay.records[i][0] else (i // 64 + 1) * 64
        at = [i for i, r in enumerate(replay.records) if r[0] == FWD and i not in headers
              and struct.unpack("<i", r[4:8])[0] > 2]
        if not at:
            continue
        ran += 1
        i = rng.choice(at)
        r = bytearray(replay.records[i])
        if route == "teams" and ran % 2 and i % 64 and replay.records[i - 1][0] and replay.records[i - 1][2] & 1:
            q = bytearray(replay.records[i - 1])
            q[2] &= ~1                                                                         # no end of the phase before
            replay.records[i - 1] = bytes(q)
        else:
            struct.pack_into("<I", r, 8, struct.unpack_from("<I", r, 8)[0] + replay.parts)     # src
            replay.records[i] = bytes(r)
        with pytest.raises(AssertionError):
            replay.run()
