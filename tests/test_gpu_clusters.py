"""GPU: runs of the bfloat16 recurrence inside a thread-block cluster (one layer of at most 512 units), at the edges
of what a cluster, a CTA and an MMA tile hold; and the grid-wide kernels that wider layers keep.
"""
import json
import os
import subprocess
import sys

import pytest

from paper_1606_03401_b200 import synth
from tests.test_gpu_variants import CHILD, ROOT
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
@pytest.mark.parametrize("hidden,batch", [(72, 9), (640, 64), (640, 20)])
def test_waits_of_both_kinds_of_runs_run_out_and_report_timeout(bit, hidden, batch):
    from paper_1606_03401_b200 import binding as B
    cfg, dp = _problem(input=40, hidden=hidden, batch=batch, readout=24, t=12)
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


def test_backward_kernels_of_wide_layers_give_the_same_bits():
    child = CHILD.replace("hidden=256", "hidden=640")
    assert child != CHILD

    def digest(env_extra):
        env = {k: v for k, v in os.environ.items() if not k.startswith("MEBPTT_")}
        env.update(env_extra)
        out = subprocess.run([sys.executable, "-c", child.format(root=ROOT)], env=env, capture_output=True, text=True, timeout=600)
        assert out.returncode == 0, out.stderr[-2000:]
        return json.loads([l for l in out.stdout.splitlines() if l.startswith("DIGEST ")][-1][len("DIGEST "):])

    base = digest({})
    assert base["msm"] == base["full"]
    assert digest({"MEBPTT_BWD_CLUSTER": "4"}) == base
