"""The push pass over blocks of 512 elements, at the sizes where it can go wrong: a last block that is shorter and alone in
its round, layers that begin or end inside a block, many layers in one block, layers of a single element, layers that
straddle two CTAs' shares.  Everything is compared bit for bit with the CPU checker."""
import pytest

import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import replay_and_compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,ppm", [
    ([1], 1_000_000),                                 # one element
    ([8 * 512 + 3], 20_000),                          # the shorter block alone in its round
    ([512, 512, 1], 30_000),                          # layers that end with a block
    ([511, 2, 511, 4 * 512, 1], 30_000),              # ... and one element before and after
    ([1] * 700 + [3_000], 500_000),                   # hundreds of layers in a block
    ([64, 576, 64, 64, 36_864, 64, 64, 147_456], 10_000),
    ([100_003, 7, 300_001, 129, 50_000], 100_000),    # several CTAs a layer, dense
])
@pytest.mark.parametrize("flags", [0, dgs.DGS_RESIDUAL_MODE])
def test_push_edges(sizes, ppm, flags):
    wl = W.custom("push", sizes, 2, 6, ppm, grad_kind="laplace")
    replay_and_compare(wl, flags=flags, compare_state_every=3)
