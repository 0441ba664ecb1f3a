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


def _refused(desc, nbytes, mode):
    try:
        return B.mebptt_plan_for_bytes(desc, nbytes, mode, include_working=True)
    except B.MebpttError as e:
        assert e.status == B.MEBPTT_ERR_BUDGET
        return None


@pytest.mark.parametrize("size,least", [
    ((2, 161, 300, 29, 20, 160, "bf16", False), 1_000_000),     # teams
    ((2, 161, 300, 29, 40, 160, "bf16", False), 1_750_000),     # teams
    ((1, 77, 200, 61, 13, 120, "fp32", False), 300_000),        # pods
    ((2, 128, 256, 128, 32, 128, "bf16", True), 1_000_000),     # pods
    ((1, 32, 64, 32, 4, 64, "fp32", False), 25_000),            # pods, one length of chunk
])
@pytest.mark.parametrize("mode", [B.MEBPTT_HSM, B.MEBPTT_MSM])
def test_a_whole_device_budget_is_met_from_a_few_states_on(size, least, mode):
    """What the operation-by-operation kernels hold beside the states was always enough for a plan; more memory
    never makes one more expensive on the same kernels, and the kernels that walk the tape come in with it."""
    desc = _problem(size)
    assert _refused(desc, least // 4, mode) is None
    seen, cheapest, nbytes = [], {}, least
    while nbytes < 200_000_000:
        plan = _refused(desc, nbytes, mode)
        assert plan is not None, nbytes
        assert B.mebptt_lstm_workspace_bytes(desc, plan) <= nbytes
        r = B.mebptt_test_route(desc, plan)
        if r["route"] != "operations":
            # room for the states, and for one more at most
            assert B.mebptt_lstm_workspace_bytes(desc, plan) - B.mebptt_lstm_working_bytes(desc, plan) > 0
        key = (r["route"], r["chunk"])
        assert plan.cost <= cheapest.get(key, plan.cost)
        cheapest[key] = plan.cost
        seen.append(r["chunk"])
        nbytes = nbytes * 7 // 6
    assert seen[0] == 0 and seen == sorted(seen) and seen[-1] == B.mebptt_test_route(desc, B.mebptt_plan(size[5], 8, mode))["chunk"]


@pytest.mark.parametrize("use_beta", [False, True])
def test_a_whole_device_budget_in_exact_sizes_is_met_too(use_beta):
    desc = _problem((2, 161, 300, 29, 40, 160, "bf16", False))
    for nbytes in (2_000_000, 5_000_000, 20_000_000, 60_000_000):
        plan = B.mebptt_plan_bytes_exact(desc, nbytes, use_beta, include_working=True)
        assert plan.sigma == 5 and B.mebptt_lstm_workspace_bytes(desc, plan) <= nbytes
    assert B.mebptt_test_route(desc, plan)["route"] == "teams"


def test_chunks_are_whole_blocks_of_sums():
    """The weight gradients are summed in blocks of a fixed number of steps: a chunk that cut one would change bits."""
    for batch in (1, 5, 13, 32, 33, 48, 100, 129, 3000):
        desc = _problem((2, 20, 40, 10, batch, 400, "fp32", False))
        blocks = next(s for s in (1, 2, 4, 8, 16, 32, 64) if s * batch >= 256 or s == 64)
        for nbytes in (10 ** 6 * k * k for k in range(1, 24, 2)):
            plan = _refused(desc, nbytes * (1 + batch // 40), B.MEBPTT_HSM)
            if plan is not None:
                assert B.mebptt_test_route(desc, plan)["chunk"] % blocks == 0
