"""GPU: the contraction's rings at their edges, against the definition in float64.

A grid of one wave takes three tiles of 64 contraction indices a stage where there are more than six of them, by one copy
where the columns are whole blocks of 64 and by several where they are not; larger grids take one a stage.  The bound is
that of the other tests of the contraction: float32 sums of K products of two standard normal values, relative to
the largest of the results.
"""
import numpy as np
import pytest

from tests.test_gpu_gemm import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a_mn,b_mn", [(False, False), (True, True), (True, False), (False, True)])
@pytest.mark.parametrize("M,N", [(128, 128), (192, 136), (72, 64)])
@pytest.mark.parametrize("K", [384, 392, 448, 512, 576, 640, 1000])
def test_stages_of_three_tiles(M, N, K, a_mn, b_mn):
    assert _run(M, N, K, a_mn, b_mn, accumulate=True, bias=not a_mn, pad=8) < 2e-6 * np.sqrt(K) + 1e-6


@pytest.mark.parametrize("M,N", [(1664, 1536), (1672, 1544)])      # 13 x 12 tiles: more than a wave
@pytest.mark.parametrize("K", [448, 456])
def test_grids_of_more_than_a_wave(M, N, K):
    for mn in (False, True):
        assert _run(M, N, K, mn, mn, accumulate=True) < 2e-6 * np.sqrt(K) + 1e-6
