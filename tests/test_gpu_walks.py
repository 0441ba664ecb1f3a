"""GPU parity of the kernels that walk a whole tape or a whole run: sizes at the edges of their tiles,
each against the fp64 oracle and bit for bit across plans."""
import pytest

from paper_1606_03401_b200 import synth
from tests.util import assert_bit_identical, assert_close_to_oracle, oracle_run

pytestmark = pytest.mark.gpu

# (type, GRU, tensor cores forbidden, sizes): layers, input, hidden, batch, t, readout
SHAPES = [
    # clusters: one CTA, ragged units and rows; several layers; the widest that fit; weights read from the L2
    ("fp32", False, False, (1, 9, 33, 2, 70, 7)),
    ("fp32", False, False, (3, 20, 61, 9, 12, 33)),
    ("fp32", True, False, (2, 65, 200, 17, 10, 5)),
    ("fp32", False, False, (1, 160, 256, 32, 9, 130)),
    ("bf16", False, False, (2, 17, 31, 3, 40, 29)),
    ("bf16", False, False, (2, 128, 256, 32, 20, 128)),
    ("bf16", True, False, (2, 33, 130, 9, 20, 70)),
    ("tf32", False, False, (1, 40, 160, 32, 20, 24)),
    # the cooperative grid: more rows than one pass takes, one row, contractions with a remainder
    ("bf16", False, False, (2, 33, 301, 40, 10, 29)),
    ("bf16", False, False, (1, 65, 515, 1, 8, 10)),
    ("bf16", False, True, (1, 64, 264, 11, 9, 40)),
    ("bf16", True, False, (1, 100, 512, 64, 8, 33)),
    ("fp32", False, False, (2, 50, 520, 70, 6, 11)),
    # persistent runs with float32 storage: both numbers of batch groups, columns padded to a block of 64
    ("tf32", False, False, (1, 24, 232, 64, 45, 40)),
    ("tf32", False, False, (1, 8, 512, 64, 20, 16)),
    ("tf32", False, False, (1, 64, 712, 32, 40, 104)),
    ("tf32", False, False, (1, 40, 1000, 32, 35, 48)),
]


@pytest.mark.parametrize("dtype,gru,forbid,size", SHAPES)
def test_walks_match_the_oracle_and_one_another(dtype, gru, forbid, size):
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    keys = ("layers", "input", "hidden", "batch", "t", "readout")
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype=dtype, **dict(zip(keys, size)), **({"cell": "gru"} if gru else {}))
    dp = H.DeviceProblem(cfg, want_dx=True, flags=B.MEBPTT_FLAG_NO_TENSOR_CORES if forbid else 0)
    full = dp.run(dp.full_memory_plan())
    assert_close_to_oracle(full, oracle_run(dp.prob), dtype, want_dx=True)
    for mode, m, beta in [("hsm", 3, 0), ("ism", 2, 0), ("msm", 9, 3), ("hsm", cfg.t, 0)]:
        plan = dp.plan(mode, m, beta=beta)
        res = dp.run(plan)
        assert res["counters"][0] == plan.cost and res["counters"][1] == cfg.t and res["counters"][3] == 0
        assert_bit_identical(res, full, want_dx=True)
