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
