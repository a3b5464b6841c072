"""The pass that folds the filed packets into a difference vector and scans it, at the sizes where it can go wrong:
vectors of one partial block, one block more or less than a group, blocks with more entries than are fetched ahead,
more packets than a warp has lanes, layers that end inside a block.  Everything is compared bit for bit with the CPU
checker."""
import pytest

import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import replay_and_compare, replay_async_and_compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,workers,ppm,away", [
    ([1], 2, 1_000_000, 0),                       # one element
    ([511], 3, 20_000, 0),                        # less than a block
    ([512], 3, 20_000, 0),
    ([4097], 3, 5_000, 0),                        # a group of blocks and one element
    ([37 * 512], 4, 500_000, 0),                  # 1024 entries a block: most are not fetched ahead
    ([9_000], 3, 400_000, 45),                    # the same, and more than 32 packets missed
    ([100, 3, 1, 409, 600, 64, 5_000], 3, 30_000, 40),   # several layers inside one block, packets beyond the first 32
    ([300_001], 5, 300, 0),                       # most blocks have no entry and a bound below the selection's
])
def test_fold_edges(sizes, workers, ppm, away):
    wl = W.custom("fold", sizes, workers, 6 * workers, ppm, grad_kind="laplace")
    last = workers - 1
    sched = [e % workers for e in range(2 * workers)]
    sched += [e % last for e in range(away)] + [last] + [e % workers for e in range(workers)]
    replay_and_compare(wl, schedule=sched, compare_state_every=0 if away else workers)
    replay_async_and_compare(wl, schedule=sched, flags=dgs.DGS_KEEP_LOCAL_MODEL)
