"""Packets of the caller's own at the server: filed in the log (any length up to the library's), scattered (longer),
between the library's own events, with the caller joining after every call or never.  Bit for bit against the CPU
checker."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import compare_state, packet_to_numpy

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("join", [True, False])
@pytest.mark.parametrize("workers", [1, 2, 5, 40])
@pytest.mark.parametrize("flags", [0, dgs.DGS_SINGLE_STREAM])
def test_foreign_packets_between_events(workers, join, flags):
    n = 40_000
    wl = W.custom("foreign", [n], workers, 1, 5_000, grad_kind="normal")       # K = 200, log slots of 256
    theta0 = wl.theta0()
    orc = oracle.Oracle.from_workload(wl, theta0=theta0)
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(theta0).to(DEV), flags=flags)
    rng = np.random.default_rng(workers)
    keep = []                                                                  # packets must outlive the enqueued work
    for e, count in enumerate([1, 200, 256, 257, 3_000, 7, 200, n, 31, 256] * 4):
        w = int(rng.integers(workers))
        idx = np.sort(rng.choice(n, count, replace=False)).astype(np.uint32)
        val = rng.standard_normal(count, dtype=np.float32)
        pair = torch.from_numpy(idx.view(np.int32)).to(DEV), torch.from_numpy(val).to(DEV)
        keep.append(pair)
        ctx.server_apply(w, dgs.dgs_packet(pair[0].data_ptr(), pair[1].data_ptr(), count))
        orc.apply(w, idx, val)
        if e % 3 == 1:
            g = rng.standard_normal(n, dtype=np.float32)
            keep.append(torch.from_numpy(g).to(DEV))
            ctx.event(w, keep[-1])
            orc.event(w, g)
        elif e % 3 == 2:
            pull = ctx.worker_pull(w)
            want = orc.pull(w)
            if join:
                gi, gv = packet_to_numpy(ctx, pull)
                assert np.array_equal(gi, want[0]) and np.array_equal(gv, want[1])
        if join:
            ctx.flush()
    assert ctx.status() == 0
    compare_state(ctx, orc, workers, False)


def test_a_packet_that_does_not_ascend_is_reported():
    n = 5_000
    ctx = dgs.Context(n, 2, 0.1, 0.9, [0], [n], [10], [10], torch.zeros(n, device=DEV))
    idx = torch.tensor([7, 1, 4000], dtype=torch.int32, device=DEV)
    val = torch.ones(3, device=DEV)
    ctx.server_apply(0, dgs.dgs_packet(idx.data_ptr(), val.data_ptr(), 3))
    assert ctx.status() != 0


@pytest.mark.parametrize("count", [3, 64, 65, 1_000])          # the library files packets of up to 64 entries here
@pytest.mark.parametrize("fault", ["none", "duplicate", "descending", "beyond"])
def test_faulty_packets_of_any_length_are_reported(count, fault):
    n = 5_000
    ctx = dgs.Context(n, 2, 0.1, 0.9, [0], [n], [10], [10], torch.zeros(n, device=DEV))
    idx = np.arange(count, dtype=np.int64) * 4
    at = count - 2                                               # the last pair, which may open a CTA's share
    if fault == "duplicate":
        idx[at + 1] = idx[at]
    elif fault == "descending":
        idx[at + 1] = idx[at] - 1
    elif fault == "beyond":
        idx[at + 1] = n
    pair = torch.from_numpy(idx.astype(np.int32)).to(DEV), torch.ones(count, device=DEV)
    ctx.server_apply(0, dgs.dgs_packet(pair[0].data_ptr(), pair[1].data_ptr(), count))
    ctx.worker_pull(0)
    assert (ctx.status() != 0) == (fault != "none")


def test_an_own_packet_waits_for_the_callers_stream():
    """The caller's stream reads theta and a difference late; an apply of the library's own packet, and the catch-up of
    a difference that it or state() needs, must not be seen there."""
    n, workers = 50_000, 2
    wl = W.custom("late", [n], workers, 1, 5_000, grad_kind="normal")
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(wl.theta0()).to(DEV))
    g = torch.from_numpy(wl.gradient(0)).to(DEV)
    theta, D1 = ctx.state(dgs.DGS_THETA), ctx.state(dgs.DGS_D, 1)
    ring = 40                                    # more packets than the log holds: worker 1's difference is caught up
    for _ in range(ring):
        pkt = ctx.worker_push(0, g)
        ctx.flush()
        torch.cuda.synchronize()
        before = theta.clone(), D1.clone()
        torch.cuda._sleep(200_000)
        late = theta.clone(), D1.clone()
        ctx.server_apply(0, pkt)
        ctx.flush()
        assert torch.equal(late[0], before[0]) and torch.equal(late[1], before[1])
        assert not torch.equal(theta, before[0])
    before = D1.clone()
    torch.cuda._sleep(200_000)
    late = D1.clone()
    ctx.state(dgs.DGS_D, 1)
    assert torch.equal(late, before) and not torch.equal(D1, before)
    assert ctx.status() == 0
