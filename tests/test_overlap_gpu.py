"""Events that overlap, at every number of workers near the number of streams: bounds are carried from the selections of
other workers whose events are still in flight.  State and packets, bit for bit against the CPU checker."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import compare_state, packet_to_numpy

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("workers", [1, 2, 3, 7, 8, 9, 10, 17])
@pytest.mark.parametrize("arrivals", ["cyclic", "uniform"])
def test_long_runs_without_a_join(workers, arrivals):
    n, events = 60_000, 96
    wl = W.custom("overlap", [n - 1_000, 1_000], workers, events, 5_000, grad_kind="normal")
    theta0 = wl.theta0()
    orc = oracle.Oracle.from_workload(wl, theta0=theta0, keep_local=True)
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(theta0).to(DEV), flags=dgs.DGS_KEEP_LOCAL_MODEL)
    rng = np.random.default_rng(workers)
    grads = [rng.standard_normal(n, dtype=np.float32) for _ in range(11)]
    on_gpu = [torch.from_numpy(g).to(DEV) for g in grads]
    torch.cuda.synchronize()
    for e in range(events):
        w = e % workers if arrivals == "cyclic" else int(rng.integers(workers))
        push, pull = ctx.event(w, on_gpu[e % 11])
        want = orc.event(w, grads[e % 11])
    for got, ref in zip((push, pull), want):
        gi, gv = packet_to_numpy(ctx, got)
        assert np.array_equal(gi, ref[0]) and np.array_equal(gv, ref[1])
    assert ctx.status() == 0
    compare_state(ctx, orc, workers, True)
