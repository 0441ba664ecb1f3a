"""Host: what the kernels that walk a whole tape need beside the states (no GPU needed)."""
import pytest

from paper_1606_03401_b200 import binding as B

# layers, input, hidden, readout, batch, t, type, GRU: problems of pods and of teams
WALKED = [
    (1, 32, 64, 32, 4, 64, "fp32", False),
    (2, 77, 200, 61, 13, 120, "fp32", False),
    (2, 128, 256, 128, 32, 128, "bf16", True),
    (2, 161, 300, 29, 20, 160, "bf16", False),
    (1, 65, 515, 10, 1, 8, "bf16", False),
]


def _problem(size):
    L, I, H, O, N, t, dtype, gru = size
    return B.make_desc(L, I, H, O, N, t, dtype, want_dx=1, flags=B.MEBPTT_FLAG_GRU if gru else 0)


@pytest.mark.parametrize("size", WALKED)
def test_weights_are_packed_in_the_order_of_the_kernel_that_runs_and_no_other(size):
    L, I, H, O, N, t, dtype, gru = size
    desc, plan = _problem(size), B.mebptt_plan(t, 8, B.MEBPTT_HSM)
    route = B.mebptt_test_route(desc, plan)
    e, S = (2 if dtype == "bf16" else 4), route["chunk"]
    # stages of a chunk, carried gradients, two cores and three states, tape
    stages = L * S * N * 4 * H * 4 + L * (S + 1) * N * H * e + S * N * O * 4
    carried = L * N * H * 4 * (1 + 2 * 4)
    states = L * N * H * (2 * (4 * e + 2 * (e + 4)) + 3 * (e + 4))
    tape = min(1 << 20, 32 * (7 * (plan.cost * L + t * (L + 2)) + 400))
    # rows padded to their kernel's tiles, units to its CTAs: a quarter and some more, of one copy of the weights
    # on pods; teams keep a transposed one besides
    weights = (L * 4 * H * (2 * H + 120) + 4 * H * max(0, I - H) + (O + 64) * (H + 104)) * e
    weights = 1.25 * weights * (1 if route["route"] == "pods" else 2)
    assert B.mebptt_lstm_working_bytes(desc, plan) <= stages + carried + states + tape + weights + 64 * 1024


@pytest.mark.parametrize("size", WALKED)
@pytest.mark.parametrize("mode,m", [(B.MEBPTT_HSM, 2), (B.MEBPTT_MSM, 9), (B.MEBPTT_ISM, 10 ** 6)])
def test_no_launch_has_more_records_than_there_is_room_for(size, mode, m):
    """A launch reads its records from a region of the workspace; whatever the region's size, they fit, and
    every operation is still there once."""
    desc, plan = _problem(size), B.mebptt_plan(size[5], m, mode)
    layers = size[0]
    for room in (0, 256, 1024, 32768):
        info, records, launches = B.mebptt_test_schedule(desc, plan, room)
        assert launches[:, 1].max() <= (room or info["room"])
        assert (launches[:, 0] + launches[:, 1]).max() <= len(records) and (launches[:, 1] % 64 == 0).all()
        assert (launches[:, 3] >= 0).sum() == -(-size[5] // info["chunk"])
        if not info["pods"]:      # (a pod's headers are records of another kind: replayed elsewhere)
            kinds = records[:, 0]
            assert (kinds == 1).sum() == plan.cost * layers and (kinds == 3).sum() == size[5] * layers


@pytest.mark.parametrize("dtype,gru", [("fp32", False), ("bf16", False), ("bf16", True)])
def test_plans_over_byte_sizes_take_the_kernels_of_other_plans(dtype, gru):
    """The unit of such a plan is any fraction of a hidden state (seventh parts among these)."""
    sigmas = set()
    plan = B.mebptt_plan(20, 5, B.MEBPTT_HSM)
    for layers in (1, 2, 3):
        for hidden in (20, 64, 100, 200, 300):
            for batch in (1, 5, 9, 20, 40, 48):
                desc = _problem((layers, 16, hidden, 8, batch, 20, dtype, gru))
                exact = B.mebptt_plan_bytes_exact(desc, 12 * B.mebptt_lstm_unit_bytes(desc))
                want, got = B.mebptt_test_route(desc, plan), B.mebptt_test_route(desc, exact)
                assert got == want and want["route"] in ("pods", "teams", "persistent"), (layers, hidden, batch)
                sigmas.add(exact.sigma)
    assert dtype == "fp32" or {2, 3, 5, 7} <= sigmas
