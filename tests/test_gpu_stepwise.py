"""GPU: every way a step can run, on problems that are known to take it.

``mebptt_test_route`` says which kernels serve a problem, and each test here asserts it: shapes move from one path
to another as paths are added, and a test that compares two ways of doing one thing would otherwise go on to
compare a third with itself.
"""
import pytest

from oracle import policy as P
from paper_1606_03401_b200 import synth
from tests.util import assert_bit_identical, assert_close_to_oracle, launches_of_a_step, oracle_run, rel_l2

pytestmark = pytest.mark.gpu

KEYS = ("layers", "input", "hidden", "readout", "batch", "t")

# type, sizes: several layers, ragged columns of tiles, batches of one to four row groups, more than two chunks
STEPWISE = [
    ("stepwise", "bf16", (2, 64, 640, 40, 64, 75)),
    ("stepwise", "bf16", (3, 24, 712, 8, 96, 50)),
    ("stepwise", "bf16", (1, 128, 1152, 64, 64, 9)),
    ("stepwise_f32", "tf32", (2, 64, 768, 40, 32, 70)),
    ("stepwise_f32", "tf32", (3, 40, 776, 24, 64, 37)),
    ("stepwise_f32", "tf32", (1, 24, 640, 8, 96, 45)),
]


def _problem(dtype, size, general=True, **kw):
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype=dtype, **dict(zip(KEYS, size)))
    return cfg, H.DeviceProblem(cfg, synth.make_problem(cfg, general=general), **kw)


def _route(dp, plan):
    from paper_1606_03401_b200 import binding as B
    return B.mebptt_test_route(dp.desc, plan)["route"]


@pytest.mark.parametrize("route,dtype,size", STEPWISE)
def test_step_by_step_paths_match_the_oracle_under_every_plan(route, dtype, size):
    """Oracle parity per tensor and per block with general biases and initial state, bit identity across plans,
    agreement with FMA kernels, and no difference without dx."""
    from paper_1606_03401_b200 import binding as B
    cfg, dp = _problem(dtype, size, want_dx=True)
    full = dp.run(dp.full_memory_plan())
    assert _route(dp, dp.full_memory_plan()) == route and full["counters"][3] == 0
    assert_close_to_oracle(full, oracle_run(dp.prob), dtype, want_dx=True)
    for mode, m, beta in [("hsm", 1, 0), ("hsm", 4, 0), ("ism", 2, 0), ("msm", 9, 0), ("msm", 13, 3)]:
        plan = dp.plan(mode, m, beta=beta)
        res = dp.run(plan)
        code = {"hsm": P.HSM, "ism": P.ISM, "msm": P.MSM}[mode]
        assert res["counters"][0] == plan.cost == P.cost(code, cfg.t, plan.m, 4, beta or None)
        assert res["counters"][1] == cfg.t and res["counters"][3] == 0
        assert_bit_identical(res, full, want_dx=True)
    from paper_1606_03401_b200 import harness as H
    slow = H.DeviceProblem(cfg, dp.prob, want_dx=True, flags=B.MEBPTT_FLAG_NO_TENSOR_CORES)
    other = slow.run(slow.full_memory_plan())
    for k in ("dW", "db", "dW_out", "db_out", "dx"):
        assert rel_l2(full[k], other[k]) < (1e-2 if dtype == "bf16" else 1e-4), k
    nodx = H.DeviceProblem(cfg, dp.prob, want_dx=False)
    assert_bit_identical(nodx.run(nodx.plan("msm", 9)), full)


@pytest.mark.parametrize("route,dtype,size", STEPWISE + [
    ("stepwise", "bf16", (2, 128, 2048, 128, 128, 19)),
    ("runs_f32", "tf32", (1, 64, 1000, 40, 32, 70)),
    ("runs_f32", "tf32", (1, 40, 512, 24, 64, 45)),
])
def test_runs_give_the_bits_of_single_operations(route, dtype, size, monkeypatch):
    """Runs of consecutive operations, a layer or a launch at a time, with what can be batched over the run batched,
    against MEBPTT_STEPWISE_PER_OP=1: long runs and short ones, with and without dx."""
    for want_dx in (True, False):
        cfg, dp = _problem(dtype, size, want_dx=want_dx)
        plans = [dp.full_memory_plan(), dp.plan("msm", 11), dp.plan("hsm", 3), dp.plan("ism", 2)]
        assert all(_route(dp, p) == route for p in plans)
        runs = [dp.run(p) for p in plans]
        monkeypatch.setenv("MEBPTT_STEPWISE_PER_OP", "1")
        single = dp.run(plans[0])
        monkeypatch.delenv("MEBPTT_STEPWISE_PER_OP")
        for p, r in zip(plans, runs):
            assert r["counters"][0] == p.cost and r["counters"][1] == cfg.t and r["counters"][3] == 0
            assert_bit_identical(r, single, want_dx=want_dx)


@pytest.mark.parametrize("route,dtype,gru,size", [
    ("persistent", "bf16", False, (1, 128, 256, 128, 64, 70)),
    ("persistent", "bf16", False, (1, 40, 640, 24, 64, 50)),
    ("stepwise", "bf16", False, (2, 64, 640, 40, 64, 75)),
    ("stepwise", "bf16", False, (2, 128, 2048, 128, 128, 19)),
    ("stepwise_f32", "tf32", False, (2, 64, 768, 40, 32, 70)),
    ("stepwise_f32", "tf32", False, (1, 24, 640, 8, 96, 45)),
    ("runs_f32", "tf32", False, (1, 64, 1000, 40, 32, 70)),
    ("pods", "fp32", False, (1, 32, 64, 32, 4, 90)),
    ("pods", "bf16", True, (2, 64, 256, 40, 32, 40)),
    ("teams", "bf16", False, (2, 40, 300, 29, 40, 70)),
    ("operations", "fp32", False, (2, 33, 96, 20, 13, 20)),
    ("operations", "bf16", False, (2, 40, 300, 29, 40, 20)),
    ("operations", "bf16", True, (2, 40, 300, 29, 40, 20)),
])
@pytest.mark.parametrize("want_dx", [False, True])
def test_launch_count_is_what_the_profiler_sees_on_every_path(route, dtype, gru, size, want_dx):
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype=dtype, **dict(zip(KEYS, size)), **({"cell": "gru"} if gru else {}))
    dp = H.DeviceProblem(cfg, want_dx=want_dx)
    plans = [dp.plan("msm", 11), dp.plan("hsm", cfg.t), dp.full_memory_plan()]
    if route == "operations":       # a budget that holds a few states beside the least working memory
        unit, nbytes = B.mebptt_lstm_unit_bytes(dp.desc), 0
        plans = []
        while len(plans) < 2:
            nbytes += 5 * unit
            try:
                plans.append(B.mebptt_plan_for_bytes(dp.desc, nbytes, B.MEBPTT_MSM, include_working=True))
            except B.MebpttError:
                pass
    for plan in plans:
        assert _route(dp, plan) == route
        res = dp.run(plan)
        assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
        made, seen = launches_of_a_step(dp, plan)
        assert seen <= made == B.mebptt_lstm_launch_count(dp.desc, plan), (plan.cost, made, seen)
