"""The finalize of a selection at the sizes where it can go wrong: lists that are ranked in shared memory, by radix
steps, or are too short (ties); layers that begin and end inside a warp's candidates; more layers than the tables in
shared memory hold; candidates that do not fit the registers.  Bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def values(kind: str, n: int) -> np.ndarray:
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n, dtype=np.float32)
    if kind == "ties":           # a handful of values: every list is too short
        x = np.round(x * 4).astype(np.float32)
    elif kind == "narrow":       # all keys within a few bins: lists of hundreds to thousands of entries
        x = (1.0 + rng.random(n, dtype=np.float32) * 2.0 ** -7).astype(np.float32)
    elif kind == "wide":         # many octaves: the k-th far above the bound
        x = np.exp(x * 8).astype(np.float32)
    elif kind == "sparse":       # fewer nonzero values than are taken
        x[rng.random(n) < 0.995] = 0.0
    return x


@pytest.mark.parametrize("kind", ["normal", "ties", "narrow", "wide", "sparse"])
@pytest.mark.parametrize("sizes,ppm", [([257], 100_000), ([65_536], 1000), ([300_001], 20_000), ([1 << 20], 400_000),
                                       ([1] * 70 + [5_000] + [33] * 40 + [100_000], 10_000), ([700] * 90, 60_000),
                                       ([400_000, 7, 300_001, 513], 500_000)])
def test_finalize_edges(sizes, ppm, kind):
    n = sum(sizes)
    ks = [max(1, s * ppm // 1_000_000) for s in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    ctx = dgs.Context(n, 1, 0.1, 0.9, off, sizes, ks, ks, torch.zeros(n, device=DEV))
    for turn in range(3):        # the first selection has nothing to go by, the others a carried bound
        x = values(kind, n) * np.float32(1.0 + 0.01 * turn)
        ctx.state_load(dgs.DGS_D, 0, torch.from_numpy(x).to(DEV))
        idx, val = (t.cpu().numpy() for t in ctx.packet(ctx.worker_pull(0)))
        want = np.concatenate([oracle.topk(x[o:o + s], k).astype(np.int64) + o for o, s, k in zip(off, sizes, ks)])
        assert np.array_equal(idx.view(np.uint32), want.astype(np.uint32)), turn
        assert np.array_equal(val.view(np.uint32), x[want].view(np.uint32)), turn
        left = ctx.state(dgs.DGS_D, 0).cpu().numpy()
        x[want] = 0.0
        assert np.array_equal(left, x), turn
    assert ctx.status() == 0


def test_barriers_that_give_up_again_and_again():
    """A selection whose barrier gave up leaves its counts behind: the lists of the later ones stay in their places, and
    the arena beside them as it was."""
    sizes = [40_000, 300, 513]
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    n, ks = sum(sizes), [400, 3, 5]
    theta0 = torch.randn(n, device=DEV)
    ctx = dgs.Context(n, 1, 0.1, 0.9, off, sizes, ks, ks, theta0, flags=dgs.DGS_TEST_STALLED_BARRIER | dgs.DGS_NO_SPECULATION)
    for turn in range(60):       # every turn has its own k-th, so that every list is another bin's
        g = torch.from_numpy(values("normal", n) * np.float32(1.3 ** (turn % 20))).to(DEV)
        ctx.worker_push(0, g)
        assert ctx.status() == dgs.DGS_ETIMEOUT
    assert torch.equal(ctx.state(dgs.DGS_THETA), theta0)
