"""The convolutional generator's kernels around the sizes where their rules change over: the tiled
convolutions (from 125,000 outputs of a middle layer) and the weight-gradient product (from 2600
positions), just below and above, and above them at the edges of the tiles (channel counts off the
groups of 8 and past 32, odd rows, rows and slices of length 1 and 2). The checks and bars are those of
the tiles' own tests: integer inputs whose sums are exact, so logits are equal bit for bit, and
gradients to 3e-2 of a layer's largest entry (one BF16 unit where an FP32 and an FP64 sum straddle a
rounding boundary)."""
import pytest

import test_gpu_cgen_tiles as tiles
from test_gpu_cgen_tiles import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

FORWARD = [((7, 6, 4), 16, 46), ((7, 6, 4), 16, 47), ((3, 10, 10), 24, 18), ((5, 1, 2), 3, 4167),
           ((4, 2, 2), 40, 196), ((30, 6, 6), 9, 13), ((5, 4, 3), 12, 174), ((1, 4, 4), 8, 977)]
GRADIENTS = [((7, 6, 4), 16, 15), ((7, 6, 4), 16, 16), ((3, 10, 10), 24, 9), ((5, 1, 2), 3, 261),
             ((30, 6, 6), 9, 3), ((1, 4, 4), 8, 163), ((3, 10, 10), 24, 18), ((4, 2, 2), 40, 196)]


@pytest.mark.parametrize("shape,C,n", FORWARD)
def test_forward_bits(env, shape, C, n):  # noqa: F811
    tiles.test_forward_bits(env, shape, C, n)


@pytest.mark.parametrize("shape,C,n", GRADIENTS)
def test_gradients(env, shape, C, n):  # noqa: F811
    tiles.test_gradients(env, shape, C, n)
