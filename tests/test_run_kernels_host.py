"""Host: what the kernels that walk runs of a recurrence rely on, at every size they take (no GPU needed)."""
import pytest

from paper_1606_03401_b200 import binding as B

SM_BYTES, CTA_RESERVED, CTA_MOST = 228 * 1024, 1024, 227 * 1024

# route, runs of few operations, widths, batch rows a cluster or group
KERNELS = [
    ("persistent", False, range(64, 513, 8), (8, 12)),     # clusters
    ("persistent", False, range(520, 1025, 8), (8, 16)),   # ring
    ("persistent", True, range(640, 1025, 128), (32,)),
    ("runs_f32", False, range(64, 1025, 8), (32,)),
]


@pytest.mark.parametrize("route,shorter,widths,rows", KERNELS)
@pytest.mark.parametrize("backward", [False, True])
def test_an_sm_has_room_for_one_cta_that_holds_tensor_memory_and_waits_for_others(route, shorter, widths, rows, backward):
    """Two such CTAs on an SM could wait for one another's columns, each kernel for its own CTA: nothing but shared
    memory keeps them apart."""
    for hidden in widths:
        for r in rows:
            dynamic = B.mebptt_test_run_smem(route, hidden, r, backward, shorter)
            assert 2 * (dynamic + CTA_RESERVED) > SM_BYTES, hidden
            assert dynamic <= CTA_MOST, hidden



@pytest.mark.parametrize("hidden,batch,t,most", [
    (520, 1, 7, 8053760), (520, 1, 100, 8120320), (520, 17, 100, 49853440), (640, 2, 7, 13720320), (776, 64, 7, 136625664),
    (1024, 1, 100, 23150592), (1024, 3, 100, 33357824), (1024, 64, 100, 184231936),
])
def test_the_ring_takes_no_more_than_its_place_in_the_workspace(hidden, batch, t, most):
    """`most`: the workspace with a stage for h_{k-1} and one for h_k, which the ring and one stage for both replace.  (So
    small a batch as 3 rows at H = 1024 fits the 32 MB of the step without allocations.)"""
    desc = B.make_desc(1, 128, hidden, 64, batch, t, "bf16")
    assert B.mebptt_lstm_workspace_bytes(desc, B.mebptt_plan(t, 8, B.MEBPTT_HSM)) <= most


# ---- the waits inside a run, replayed with one warp as late as can be ---------------------------------------------------
# Barriers are waited for by the parity of a phase: whoever comes when the phase after that is over as well waits for good,
# or (two phases on) takes the accumulators of another step.
# Here every warp of a group of CTAs is a generator that yields what it waits for; one warp goes on only when nobody else can.

class Barrier:
    def __init__(self, count):
        self.count = self.pending = count
        self.phases, self.seen = 0, set()

    def arrive(self, who):
        assert who not in self.seen, ("twice in a phase", who)
        self.seen.add(who)
        self.pending -= 1
        if self.pending == 0:
            self.phases, self.pending, self.seen = self.phases + 1, self.count, set()

    def over(self, phase):
        return lambda: self.phases == phase + 1


def _replay(agents, late):
    """True if every agent gets to its end, `late` being held back whenever another can go on."""
    waits = {k: (lambda: True) for k in agents}
    while waits:
        moved = False
        for k in list(waits):
            if k == late:
                continue
            while k in waits and waits[k]():
                moved = True
                nxt = next(agents[k], None)
                if nxt is None:
                    del waits[k]
                else:
                    waits[k] = nxt
        if not moved:
            if late not in waits or not waits[late]():
                return False
            nxt = next(agents[late], None)
            if nxt is None:
                del waits[late]
            else:
                waits[late] = nxt
    return True


def _forward(hidden, n, waited, ring):
    """fwd_run_cluster, or fwd_run_ring (accumulators and operands twice, states polled by warps of their own)."""
    ctas, agents, sent = -(-hidden // 32), {}, {}
    sends = [(c, w) for c in range(ctas) for w in range(4) if 32 * c + 8 * w < waited]
    acc = [[Barrier(1) for _ in range(2 if ring else 1)] for _ in range(ctas)]
    full = [[Barrier(4 if ring else 1 + len(sends)) for _ in range(2)] for _ in range(ctas)]

    def phase(i):
        return (i & 1, i >> 1) if ring else (0, i)

    def mma(c):
        if not ring:
            for b in (1, 0)[:n - 1]:
                full[c][b].arrive("expect")
        for i in range(n):
            b = i & 1
            if ring:
                yield full[c][b].over(i >> 1)
            elif i > 0:
                yield full[c][b].over((i - 1) >> 1)
            acc[c][phase(i)[0]].arrive("mma")
            if not ring and i >= 1 and i + 2 < n:
                full[c][b].arrive("expect")

    def poll(c, p):                          # (a fourth of the units each: all have some)
        for i in range(n):
            mine = [(i, m) for j, m in enumerate(sends) if j % 4 == p]
            yield lambda: i == 0 or all(s in sent for s in mine)
            full[c][i & 1].arrive(p)

    def gates(c, w):
        for i in range(n):
            b, p = phase(i)
            yield acc[c][b].over(p)
            if (c, w) in sends:
                sent[i + 1, (c, w)] = True
                if not ring and i + 1 < n:
                    for peer in range(ctas):
                        full[peer][(i + 1) & 1].arrive((c, w))

    for c in range(ctas):
        agents["mma", c] = mma(c)
        for p in range(4 if ring else 0):
            agents["poll", c, p] = poll(c, p)
        for w in range(4):
            agents["gates", c, w] = gates(c, w)
    return agents


def _backward(hidden, n, waited):
    """bwd_run_ring: clusters of four share the contraction, CTA r of each taking dz of a quarter of the CTAs."""
    per = -(-hidden // 128)
    ctas, agents, sent = 4 * per, {}, {}
    sends = [(c, w) for c in range(ctas) for w in range(4) if 32 * c + 8 * w < waited]
    acc, zfull, full, inready, used = ([[Barrier(k) for _ in range(2)] for _ in range(ctas)] for k in (1, 1, 5, 1, 4))

    def mma(c):
        full[c][0].arrive("expect")
        full[c][1].arrive("expect")
        for i in range(n):
            yield zfull[c][i & 1].over(i >> 1)
            acc[c][i & 1].arrive("mma")

    def poll(c):
        quarter = [m for m in sends if m[0] // per == c % 4]
        for i in range(n):
            yield lambda: all((i, m) in sent for m in quarter)
            zfull[c][i & 1].arrive("poll")

    def fill(c):
        for i in range(min(2, n)):
            inready[c][i].arrive("fill")
        for i in range(n):
            yield used[c][i & 1].over(i >> 1)
            if i >= 1 and i + 1 < n:
                full[c][(i + 1) & 1].arrive("expect")
            if i + 2 < n:
                inready[c][i & 1].arrive("fill")

    def gates(c, w):
        to = c // 4 * 4 + w
        yield inready[c][0].over(0)
        for i in range(n):
            if i > 0:
                yield full[c][(i - 1) & 1].over((i - 1) >> 1)
            sent[i, (c, w)] = True
            used[c][i & 1].arrive((c, w))
            if i + 1 < n:
                yield inready[c][(i + 1) & 1].over((i + 1) >> 1)
            yield acc[c][i & 1].over(i >> 1)
            full[to][i & 1].arrive((c, w))
        yield full[c][(n - 1) & 1].over((n - 1) >> 1)

    for c in range(ctas):
        agents["mma", c], agents["poll", c], agents["fill", c] = mma(c), poll(c), fill(c)
        for w in range(4):
            agents["gates", c, w] = gates(c, w)
    return agents


def _agents(backward, hidden, waited):
    return _backward(hidden, 6, waited) if backward else _forward(hidden, 6, waited, hidden > 512)


WIDTHS = [(False, h) for h in (64, 72, 104, 264, 312, 504, 520, 552, 648, 1000)] + [(True, h) for h in (520, 544, 552, 640, 648, 776, 1000)]


@pytest.mark.parametrize("backward,hidden", WIDTHS)
def test_no_warp_of_a_run_can_come_too_late_for_a_wait(backward, hidden):
    waited, last = B.mebptt_test_run_units(backward, hidden), -(-hidden // (128 if backward else 32)) * (4 if backward else 1)
    for late in _agents(backward, hidden, waited):
        if late[1] in (0, last // 2) or late[1] >= last - 4:
            assert _replay(_agents(backward, hidden, waited), late), late


@pytest.mark.parametrize("backward,hidden,stuck", [
    (False, 72, [(2, 1), (2, 2), (2, 3)]),
    (False, 520, [(16, 1), (16, 2), (16, 3)]),
    (True, 520, [(c, w) for c in (16, 17, 18) for w in (1, 2, 3)]),   # (CTA 19 takes the dz of 16, whose sums need what all of 17 send)
])
def test_the_replay_notices_warps_that_nobody_waits_for(backward, hidden, stuck):
    """Were only units that exist waited for, warps without any could miss a phase: those that send partial sums to a CTA
    without units as well."""
    gates = [k for k in _agents(backward, hidden, hidden) if k[0] == "gates"]
    assert [k[1:] for k in gates if not _replay(_agents(backward, hidden, hidden), k)] == stuck


def test_every_warp_that_polls_a_part_of_a_step_has_something_to_wait_for():
    """Four warps poll each part in turns of pieces of eight units: a warp without any would run ahead of the others."""
    for hidden in range(264, 1025, 8):               # (up to 512 where a device has no clusters for them)
        first, waited = B.mebptt_test_ring_first_part(hidden), B.mebptt_test_run_units(False, hidden)
        for pieces in (first // 8, (waited - first) // 8):
            for in_hand in (2, 4):                   # pieces a warp has at a time: 16 rows, 8 rows
                assert 3 * in_hand < pieces <= 64, hidden
        quarter = -(-hidden // 128) * 16             # backward, pieces of two units: in halves
        for in_hand in (2, 4):
            assert 3 * in_hand < quarter // 2 <= 64, hidden


# ---- the barrier that dz crosses in backward runs inside a cluster, when a wait has run out ------------------------------
# bar.sync and bar.arrive count warps, not which, and have no limit: a warp that comes twice takes another's place, and
# whoever is left waits for good.

def _one_cta(n, failure, over_early):
    """Warps of bwd_run_cluster in one CTA: at step `failure` what peers push never comes.  over_early: the wait for the MMAs ends
    when another wait has run out (the model notices what that does); otherwise with the MMAs alone."""
    state = {"failed": False, "here": 0, "crossed": 0, "mma": 0}
    COUNT = 6

    def cross(name):
        state["here"] += 1
        if state["here"] == COUNT:
            state["here"], state["crossed"] = 0, state["crossed"] + 1

    def gates(w):
        for i in range(n):
            if i > 0 and i - 1 >= failure:
                yield lambda: True                       # (polls: others may go first)
                state["failed"] = True
            cross(w)
            yield lambda: state["mma"] > i or (over_early and state["failed"])

    def syncs(name):
        for i in range(n):
            cross(name)
            turn = state["crossed"] if state["here"] else state["crossed"] - 1
            yield lambda: state["crossed"] > turn
            if name == "mma":
                state["mma"] += 1

    agents = {("gates", w): gates(w) for w in range(4)}
    agents["mma"], agents["io"] = syncs("mma"), syncs("io")
    return agents


@pytest.mark.parametrize("failure", [0, 1, 2])
def test_warps_cross_the_barrier_of_a_failed_backward_run_together(failure):
    for late in list(_one_cta(5, failure, False)):
        assert _replay(_one_cta(5, failure, False), late), late


def test_a_wait_for_products_that_ends_early_would_leave_warps_in_the_barrier():
    assert not all(_replay(_one_cta(5, 0, True), late) for late in list(_one_cta(5, 0, True)))
