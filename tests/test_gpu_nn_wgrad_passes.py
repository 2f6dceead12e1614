"""The weight-gradient contraction where a block takes more than one group of
32 pixels (the grid has 304 blocks): the registers' prefetch, the shared
memory's reuse and the sums across groups, against the FP64 oracle."""

import pytest

from tests import test_gpu_nn_wgrad as W

pytestmark = pytest.mark.gpu


# pixels a parity: 17280 (two groups a block, a part-full last round) and 9744
# (one more group than blocks, half full)
@pytest.mark.parametrize("dims,Ls,nrhs", [((6, 4, 4, 4), 10, 3), ((2, 4, 2, 14), 14, 2)])
def test_several_groups_a_block(dims, Ls, nrhs):
    W.test_ragged_pixel_counts(dims, Ls, nrhs)
