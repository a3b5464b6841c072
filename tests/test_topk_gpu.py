"""dgs_topk_encode_static at the sizes where its one kernel can go wrong: fewer elements than a warp, one element more
or less than a cluster size takes, samples that say nothing about the vector, lists that overflow, ties across the
CTAs of the cluster.  Index sets and value bits must equal the CPU checker's selection."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def vector(kind: str, n: int) -> np.ndarray:
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n, dtype=np.float32)
    if kind == "equal":
        x[:] = -2.5
    elif kind == "two":          # most elements tie at the boundary
        x[:] = np.where(rng.random(n) < 0.3, 1.0, -1.0 - 2.0 ** -20).astype(np.float32)
    elif kind == "few":          # fewer nonzero entries than are taken
        x[rng.random(n) < 0.999] = 0.0
    elif kind in ("hidden", "shown"):   # large only where the kernel takes no sample, or only where it takes one
        m = min(n, 1024)
        s = (np.arange(m, dtype=np.uint64) * n // m).astype(np.int64)
        x[s] *= np.float32(1e4 if kind == "shown" else 1e-4)
    elif kind == "sorted":       # a part of the vector holds all that is large: lists of some warps fill up
        x = np.sort(np.abs(x))
    elif kind == "zero":
        x[:] = 0.0
    elif kind == "corner":       # everything large lies together
        x[: n // 300 + 1] *= np.float32(1e4)
    return x


@pytest.mark.parametrize("n", [1, 31, 33, 4096, 4097, 65_535, 131_073, 1 << 18, (1 << 18) + 1, (1 << 20) - 1, 1 << 20])
@pytest.mark.parametrize("kind", ["normal", "equal", "two", "few", "hidden", "shown", "sorted", "zero", "corner"])
def test_static_selection_edges(n, kind):
    x = vector(kind, n)
    xd = torch.empty(n + 1, device=DEV)[n % 2:][:n]      # odd lengths also start off a 16-byte boundary
    xd.copy_(torch.from_numpy(x))
    st = torch.cuda.current_stream().cuda_stream
    for k in sorted({1, max(1, n // 1000), max(1, n // 10), n}):
        idx = torch.full((k,), -1, dtype=torch.int32, device=DEV)
        val = torch.zeros(k, device=DEV)
        dgs.dgs_topk_encode_static(xd.data_ptr(), n, k, idx.data_ptr(), val.data_ptr(), st)
        assert dgs.dgs_topk_encode_static_status(st) == 0
        want = oracle.topk(x, k)
        assert np.array_equal(idx.cpu().numpy().view(np.uint32), want.astype(np.uint32)), k
        assert np.array_equal(val.cpu().numpy().view(np.uint32), x[want].view(np.uint32)), k
