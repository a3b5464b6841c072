"""Loading state between events that nobody has waited for: the copy has to come after the work in flight on that vector
and before everything enqueued later, and packets filed before a load do not belong to the loaded difference."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import compare_state

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("workers", [1, 3, 9])
def test_loads_between_events_in_flight(workers):
    n = 200_000
    wl = W.custom("load", [n], workers, 1, 5_000, grad_kind="normal")
    theta0 = wl.theta0()
    orc = oracle.Oracle.from_workload(wl, theta0=theta0, keep_local=True)
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(theta0).to(DEV), flags=dgs.DGS_KEEP_LOCAL_MODEL)
    rng = np.random.default_rng(workers)
    kinds = [(dgs.DGS_D, oracle.D), (dgs.DGS_THETA, oracle.THETA), (dgs.DGS_THETA_LOCAL, oracle.THETA_LOCAL), (dgs.DGS_U, oracle.U)]
    grads = []
    for e in range(24):
        w = int(rng.integers(workers))
        g = rng.standard_normal(n, dtype=np.float32)
        grads.append(torch.from_numpy(g).to(DEV))
        ctx.event(w, grads[-1])
        orc.event(w, g)
        if e % 2:
            gpu, cpu = kinds[(e // 2) % 4]
            q = int(rng.integers(workers))
            x = rng.standard_normal(n, dtype=np.float32)
            ctx.state_load(gpu, q, torch.from_numpy(x).to(DEV))      # (freed at once: the copy is on the caller's stream)
            ctypes.memmove(orc.state(cpu, q).ctypes.data, x.ctypes.data, x.nbytes)   # (the view is read-only)
    assert ctx.status() == 0
    compare_state(ctx, orc, workers, True)
