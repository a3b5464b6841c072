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


def test_loads_from_the_librarys_own_vectors():
    """The model copied into a worker's local model, or another worker's, while events that change them are in flight."""
    n, workers = 400_000, 6
    wl = W.custom("own", [n], workers, 1, 5_000, grad_kind="normal")
    theta0 = wl.theta0()
    orc = oracle.Oracle.from_workload(wl, theta0=theta0, keep_local=True)
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(theta0).to(DEV), flags=dgs.DGS_KEEP_LOCAL_MODEL)
    theta, local = ctx.state(dgs.DGS_THETA), [ctx.state(dgs.DGS_THETA_LOCAL, q) for q in range(workers)]
    grads = []
    for e in range(60):
        g = np.random.default_rng(e).standard_normal(n, dtype=np.float32)
        grads.append((g, torch.from_numpy(g).to(DEV)))
    torch.cuda.synchronize()
    for e, (g, gd) in enumerate(grads):
        w = e % workers
        ctx.event(w, gd)
        orc.event(w, g)
        if e % 4 == 3:
            q = (e // 4) % workers
            from_model = (e // 4) % 2 == 0
            ctx.state_load(dgs.DGS_THETA_LOCAL, q, theta if from_model else local[w])
            src = orc.state(oracle.THETA, 0) if from_model else orc.state(oracle.THETA_LOCAL, w)
            src = src.copy()
            ctypes.memmove(orc.state(oracle.THETA_LOCAL, q).ctypes.data, src.ctypes.data, src.nbytes)
    assert ctx.status() == 0
    compare_state(ctx, orc, workers, True)


def test_event_host_completes_what_was_enqueued_before():
    """After dgs_event_host the host may read anything, without a join: here the packets of the events before it."""
    n, workers = 3_000_000, 8
    wl = W.custom("host", [n], workers, 1, 5_000, grad_kind="normal")
    orc = oracle.Oracle.from_workload(wl)
    ctx = dgs.Context.from_workload(wl, flags=dgs.DGS_HOST_IO)
    g = np.random.default_rng(1).standard_normal(n, dtype=np.float32)
    gd, gh = torch.from_numpy(g).to(DEV), torch.from_numpy(g).pin_memory()
    side = torch.cuda.Stream()                       # not the caller's: ordered by the host alone
    torch.cuda.synchronize()
    for turn in range(4):
        pulls = [ctx.event(w, gd)[1] for w in range(1, workers)]
        ctx.event_host(0, gh)
        with torch.cuda.stream(side):
            got = [(ctx._view(p.idx, p.count, torch.int32).cpu().numpy().view(np.uint32),
                    ctx._view(p.val, p.count, torch.float32).cpu().numpy()) for p in pulls]
        for w, (gi, gv) in enumerate(got, start=1):
            wi, wv = orc.event(w, g)[1]
            assert np.array_equal(gi, wi) and np.array_equal(gv, wv), (turn, w)
        orc.event(0, g)
    assert ctx.status() == 0
