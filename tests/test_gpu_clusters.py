"""GPU: runs of the bfloat16 recurrence of one layer -- inside a thread-block cluster up to 512 units, through a ring in
the L2 and, for short runs, by the grid-wide kernels beyond -- at the edges of what a cluster, a CTA and an MMA tile hold.
"""
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1606_03401_b200 import synth
from tests.util import assert_bit_identical, assert_close_to_oracle, oracle_run

pytestmark = pytest.mark.gpu


def _problem(**size):
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c2"], **size)
    dp = H.DeviceProblem(cfg, synth.make_problem(cfg, general=True), want_dx=True)
    assert B.mebptt_test_route(dp.desc, dp.full_memory_plan())["route"] == "persistent"
    return cfg, dp


@pytest.mark.parametrize("hidden,batch", [
    (64, 1), (64, 64),          # two CTAs; one row, eight clusters
    (72, 9),                    # three CTAs, the last with 8 units; two clusters, the second with one row
    (104, 8), (136, 7),         # half an MMA slice of columns left over; a second tile of columns of dh
    (264, 33), (312, 46),       # 9 and 10 CTAs
    (496, 24), (504, 64),       # 16 CTAs, the last with half and with three quarters of its units
    (512, 64), (512, 48),
    # wider: 17 CTAs forward and 24 backward, a part of the contraction of 32 columns; 24 and 24; 25 and 32
    (520, 9), (640, 64), (768, 16), (776, 33),
    (1000, 20), (1024, 64), (1024, 1),
    (1024, 40), (1024, 41),     # the last group of 16 rows has 8, and 9
    (520, 1), (776, 3), (640, 4),              # up to three rows the ring lies beside the input projections
])
def test_clusters_match_the_oracle_and_every_plan_gives_the_same_bits(hidden, batch):
    cfg, dp = _problem(input=40, hidden=hidden, batch=batch, readout=24, t=41)
    full = dp.run(dp.full_memory_plan())
    assert full["counters"][3] == 0
    assert_close_to_oracle(full, oracle_run(dp.prob), "bf16", want_dx=True)
    # runs of one, two and many operations, leaves in batches and alone
    for mode, m, beta in [("hsm", 1, 0), ("hsm", 5, 0), ("hsm", cfg.t, 0), ("ism", 2, 0), ("msm", 9, 0), ("msm", 30, 3)]:
        plan = dp.plan(mode, m, beta=beta)
        res = dp.run(plan)
        assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
        assert_bit_identical(res, full, want_dx=True)


@pytest.mark.parametrize("bit", [1, 2])
@pytest.mark.parametrize("hidden,batch,t", [(72, 9, 12), (640, 64, 12), (640, 20, 12), (640, 64, 2)])   # clusters, ring, short runs
def test_waits_of_all_kinds_of_runs_run_out_and_report_timeout(bit, hidden, batch, t):
    from paper_1606_03401_b200 import binding as B
    cfg, dp = _problem(input=40, hidden=hidden, batch=batch, readout=24, t=t)
    plan = dp.full_memory_plan()
    clean = dp.run(plan)
    assert clean["counters"][3] == 0
    try:
        B.mebptt_test_wait_fault(bit)
        assert dp.run(plan)["counters"][3] == B.MEBPTT_ERR_TIMEOUT
    finally:
        B.mebptt_test_wait_fault(0)
    again = dp.run(plan)
    assert again["counters"][3] == 0 and again["counters"][1] == cfg.t
    assert_bit_identical(again, clean, want_dx=True)


@pytest.mark.parametrize("hidden", [256, 264, 520, 640])
@pytest.mark.parametrize("where,value", [("x", np.nan), ("x", np.inf), ("targets", np.inf), ("targets", np.nan), ("h0", None), ("c0", np.inf)])
def test_values_that_are_not_finite_pass_through_runs(hidden, where, value):
    """A ring's words of ones mean that nothing is there: no NaN that a step makes may look like that, or its wait runs out.
    One place of one batch row has the value (h0: the NaN whose bits are ones); of the others nothing changes."""
    import torch
    cfg, dp = _problem(input=40, hidden=hidden, batch=64, readout=24, t=41)
    clean = dp.run(dp.full_memory_plan())
    row, v = 11, dp.dev[where]
    at = v.view(cfg.t, cfg.batch, -1)[20, row] if where in ("x", "targets") else v.view(cfg.batch, -1)[row]
    if value is None:
        at.view(torch.int16)[2:4] = -1
    else:
        at[3] = value
    others = np.arange(cfg.batch) != row
    first = None
    for plan in (dp.full_memory_plan(), dp.plan("msm", 9), dp.plan("hsm", 1)):
        res = dp.run(plan)
        assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
        assert not np.isfinite(res["dW"]).all()
        dx, want = (r["dx"].reshape(cfg.t, cfg.batch, -1) for r in (res, clean))
        assert np.array_equal(dx[:, others], want[:, others])
        first = first or res
        for k in ("loss", "dW", "db", "dW_out", "db_out", "dx"):
            assert np.array_equal(res[k], first[k], equal_nan=True), k

def test_short_and_long_runs_of_wide_layers_give_the_same_bits():
    """Runs of few operations take other kernels: plans whose runs are all short, all long and mixed."""
    for size in (dict(hidden=640, batch=64), dict(hidden=1024, batch=37)):
        cfg, dp = _problem(input=40, readout=24, t=36, **size)
        full = dp.run(dp.full_memory_plan())
        for plan in (dp.plan("hsm", 1), dp.plan("ism", 2), dp.plan("ism", 4), dp.plan("msm", 13)):
            res = dp.run(plan)
            assert res["counters"][0] == plan.cost and res["counters"][3] == 0
            assert_bit_identical(res, full, want_dx=True)


@pytest.mark.parametrize("sizes", [(520, 256), (512, 64), (256, 1024)])
def test_steps_of_two_widths_on_two_streams_do_not_wait_for_one_another(sizes):
    """Kernels that hold tensor memory while their CTAs wait for one another, of two steps at a time."""
    import torch
    problems = [_problem(input=40, hidden=h, batch=64, readout=24, t=90)[1] for h in sizes]
    plans = [dp.full_memory_plan() for dp in problems]
    alone = [dp.run(p) for dp, p in zip(problems, plans)]
    streams = [torch.cuda.Stream() for _ in problems]
    torch.cuda.synchronize()
    for turn in range(6):
        for i in (0, 1) if turn % 2 else (1, 0):
            with torch.cuda.stream(streams[i]):
                problems[i].enqueue(plans[i])
    torch.cuda.synchronize()
    for dp, want in zip(problems, alone):
        res = {k: v.cpu().numpy() for k, v in dp.out.items()}
        res["loss"] = float(res["loss"][0])
        assert res["counters"][3] == 0
        assert_bit_identical(res, want, want_dx=True)


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, {root!r})
from tests import test_gpu_clusters as T
T.smaller_device({hidden}, {batch})
"""


def smaller_device(hidden, batch):
    """In a process of its own, whose environment says what the device has room for."""
    cfg, dp = _problem(input=40, hidden=hidden, batch=batch, readout=24, t=41)
    full = dp.run(dp.full_memory_plan())
    assert full["counters"][1] == cfg.t and full["counters"][3] == 0
    assert_close_to_oracle(full, oracle_run(dp.prob), "bf16", want_dx=True)
    for mode, m in [("hsm", 1), ("hsm", 5), ("ism", 2), ("msm", 9)]:
        plan = dp.plan(mode, m)
        res = dp.run(plan)
        assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
        assert_bit_identical(res, full, want_dx=True)
    print("BITS", _bits(full))


def _bits(res):
    return hashlib.sha256(b"".join(res[k].tobytes() for k in ("dW", "db", "dW_out", "db_out", "dx"))).hexdigest()


@pytest.mark.parametrize("hidden,batch,env,same", [
    # no clusters of more than eight CTAs: the ring, without a place of its own, in two parts of 2 and 3, 3 and 4, 4 and 4 blocks
    (264, 33, {"MEBPTT_RUN_CLUSTER": "8"}, False),
    (392, 9, {"MEBPTT_RUN_CLUSTER": "8"}, False),
    (512, 64, {"MEBPTT_RUN_CLUSTER": "8"}, False),
    # fewer SMs than the groups of a batch take: the groups, or the clusters, take turns
    (640, 64, {"MEBPTT_RUN_SMS": "40"}, True),
    (1024, 41, {"MEBPTT_RUN_SMS": "70"}, True),
    (512, 64, {"MEBPTT_RUN_CLUSTER": "8", "MEBPTT_RUN_SMS": "20"}, False),
])
def test_a_device_with_room_for_less_takes_other_kernels_or_turns(hidden, batch, env, same):
    out = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, hidden=hidden, batch=batch)], env={**os.environ, **env},
                         capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    if same:
        _, dp = _problem(input=40, hidden=hidden, batch=batch, readout=24, t=41)
        assert out.stdout.split()[-1] == _bits(dp.run(dp.full_memory_plan()))
