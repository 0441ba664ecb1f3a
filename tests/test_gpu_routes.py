"""GPU: which kernels serve a problem is settled by its descriptor: not by the plan, nor by the
device or there being one."""
import json
import os
import subprocess
import sys

import pytest

from paper_1606_03401_b200 import synth
from tests.util import assert_bit_identical, assert_close_to_oracle, oracle_run

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
sys.path.insert(0, {root!r})
from paper_1606_03401_b200 import binding as B
if {device}:
    import torch
    torch.zeros(1, device="cuda:0")
out = []
for dtype in ("fp32", "bf16"):
    for layers in (1, 2, 3):
        for hidden in (24, 64, 100, 130, 200, 256, 300, 520):
            for batch in (1, 3, 17, 33, 36, 64, 70, 140):
                for flags in (0, B.MEBPTT_FLAG_GRU):
                    desc = B.make_desc(layers, 40, hidden, 24, batch, 12, dtype, flags=flags)
                    plan = B.mebptt_plan(12, 5, B.MEBPTT_HSM)
                    r = B.mebptt_test_route(desc, plan)
                    out.append([r["route"], r["chunk"], r["ctas"], r["rows"], B.mebptt_lstm_launch_count(desc, plan),
                                B.mebptt_lstm_workspace_bytes(desc, plan)])
print("ROUTES " + json.dumps(out))
"""


def _routes(device):
    env = dict(os.environ)
    if not device:
        env["CUDA_VISIBLE_DEVICES"] = ""
    out = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, device=device)], env=env, capture_output=True,
                         text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-2000:]
    return json.loads([l for l in out.stdout.splitlines() if l.startswith("ROUTES ")][-1][len("ROUTES "):])


def test_a_count_without_a_device_is_that_of_the_device():
    with_device, without = _routes(True), _routes(False)
    assert with_device == without
    assert {r[0] for r in without} >= {"pods", "teams", "persistent"}


@pytest.mark.parametrize("size,alpha", [
    (dict(input=16, hidden=128, batch=1024, t=1100, readout=8), 4),              # of all pods together
    (dict(layers=3, input=16, hidden=256, batch=8, t=6000, readout=8), 64),      # of one pod (slots far larger than a state)
])
def test_states_past_4_gib_take_the_same_kernels_and_give_the_same_bits(size, alpha):
    """Full memory keeps more than 4 GiB of states here, which 32-bit offsets do not reach; a tight plan keeps little."""
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c1"], **size)
    dp = H.DeviceProblem(cfg, want_dx=True)
    tight, full = dp.plan("hsm", 40), dp.plan("ism", cfg.t, alpha=alpha)
    assert B.mebptt_lstm_workspace_bytes(dp.desc, full) > (4 << 30) + B.mebptt_lstm_working_bytes(dp.desc, full)
    assert B.mebptt_test_route(dp.desc, full) == B.mebptt_test_route(dp.desc, tight)
    assert B.mebptt_test_route(dp.desc, full)["route"] == "pods"
    want = dp.run(tight)
    got = dp.run(full)
    assert got["counters"][0] == cfg.t and got["counters"][3] == 0 and want["counters"][3] == 0
    assert_bit_identical(got, want, want_dx=True)


@pytest.mark.parametrize("size,gru,sigma,route", [
    (dict(layers=2, input=161, hidden=300, batch=40, t=24, readout=29), False, 5, "teams"),
    (dict(layers=1, input=16, hidden=200, batch=40, t=30, readout=8), True, 2, "pods"),
    (dict(layers=2, input=16, hidden=100, batch=40, t=30, readout=8), True, 5, "pods"),
    (dict(layers=3, input=16, hidden=64, batch=9, t=40, readout=8), False, 7, "pods"),
    (dict(layers=3, input=16, hidden=200, batch=40, t=20, readout=8), True, 2, "teams"),
])
def test_plans_in_fractions_of_a_hidden_state_give_the_bits_of_other_plans(size, gru, sigma, route):
    """Locations of such a plan are no whole blocks of a group's states."""
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype="bf16", **size, **({"cell": "gru"} if gru else {}))
    dp = H.DeviceProblem(cfg, want_dx=True)
    full = dp.run(dp.full_memory_plan())
    for units in (4, 11):
        for use_beta in (False, True):
            plan = B.mebptt_plan_bytes_exact(dp.desc, units * B.mebptt_lstm_unit_bytes(dp.desc), use_beta)
            assert plan.sigma == sigma and B.mebptt_test_route(dp.desc, plan)["route"] == route
            res = dp.run(plan)
            assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
            assert_bit_identical(res, full, want_dx=True)


@pytest.mark.parametrize("dtype,gru,size", [
    ("fp32", False, dict(layers=2, input=33, hidden=96, batch=13, t=150, readout=20)),     # pods, a ragged last chunk
    ("bf16", True, dict(layers=2, input=64, hidden=256, batch=32, t=90, readout=40)),      # pods, tensor cores
    ("bf16", False, dict(layers=2, input=40, hidden=300, batch=40, t=70, readout=29)),     # teams, 2048 rows no whole chunk
    ("fp32", False, dict(layers=2, input=24, hidden=520, batch=300, t=14, readout=16)),    # teams, a step a block
])
def test_whole_device_budgets_shorten_chunks_without_a_change_in_a_bit(dtype, gru, size):
    """A budget that counts the working memory cuts the staged chunks short, and at last the kernels that need
    any: every length of chunk gives the bits of the ordinary plan, the operations those of one another and
    both the oracle's gradients."""
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype=dtype, **size, **({"cell": "gru"} if gru else {}))
    dp = H.DeviceProblem(cfg, want_dx=True)
    ref = oracle_run(dp.prob)
    ordinary = dp.plan("msm", 12)
    full = dp.run(ordinary)
    assert_close_to_oracle(full, ref, dtype, want_dx=True)
    route, nbytes = B.mebptt_test_route(dp.desc, ordinary), 4 * B.mebptt_lstm_workspace_bytes(dp.desc, ordinary)
    seen, alone = {}, []
    while True:
        try:
            plan = B.mebptt_plan_for_bytes(dp.desc, nbytes, B.MEBPTT_MSM, include_working=True)
        except B.MebpttError:
            break
        r = B.mebptt_test_route(dp.desc, plan)
        if seen.setdefault((r["route"], r["chunk"]), 0) < 2:
            seen[r["route"], r["chunk"]] += 1
            dp._ws = None                       # exactly the workspace that was asked for
            res = dp.run(plan)
            assert dp._ws.numel() <= nbytes
            assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
            if r["route"] == route["route"]:
                assert_bit_identical(res, full, want_dx=True)
            else:
                alone.append(res)
                assert_close_to_oracle(res, ref, dtype, want_dx=True)
                assert_bit_identical(res, alone[0], want_dx=True)
        nbytes = nbytes * 4 // 5
    assert len(alone) == 2 and (route["route"], route["chunk"]) in seen and len(seen) >= 3, seen
