"""FP64 wavelet levels at the sides where the rules of their tiles change, as in
test_gpu_levels.py: plain analysis in tiles of 8 (subbands below 256), of 16
(272 = 16 x 17, 400) and wide (8 bases of 768), synthesis in tiles of 32 (from
512 blocks on), and level 1 summed over the bases tile by tile (from some 218
tiles on: 480 has 225, with 448 just below)."""
import pytest

import test_gpu_levels as levels
from test_gpu_levels import ms  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,J", [(448, 3), (544, 1), (800, 2), (1536, 1)])
def test_transforms(ms, N, J):  # noqa: F811
    levels.test_transforms_on_odd_coarse_levels(ms, N, J, "fp64", 1e-12)


@pytest.mark.parametrize("N,J,M", [(448, 1, 8), (480, 4, 8), (512, 2, 3), (768, 3, 1),
                                   (1056, 1, 5)])
def test_synthesis(ms, N, J, M):  # noqa: F811
    levels.test_synthesis_sum_over_bases(ms, N, J, M, "fp64", 1e-12)
