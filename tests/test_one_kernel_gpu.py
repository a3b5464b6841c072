"""Selections of short vectors, whose pass and finalize are one kernel beside other events (and for a pull of one layer also
alone), in turn with those that are two: at the smallest sizes, at the longest short vector and one element more.  State and
packets, bit for bit against the CPU checker."""
import ctypes
import time

import numpy as np
import pytest
import torch

import oracle
import paper_1910_10929_b200 as dgs
import workloads as W
from _replay import bits, compare_state, packet_to_numpy

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LONGEST = 3 << 19


@pytest.mark.parametrize("sizes,workers,ppm,join", [
    ([1], 3, 1_000_000, 3),
    ([513], 4, 20_000, 1),
    ([64 * 8 * 512 + 1], 5, 30_000, 4),               # a block more than one for every warp
    ([70_001, 3, 500, 9_000], 3, 10_000, 5),
    ([1] * 400 + [20_000], 4, 600_000, 7),            # more layers than a CTA's table in shared memory holds
    ([LONGEST], 3, 2_000, 4),
    ([LONGEST + 1], 3, 2_000, 4),
    ([1 << 19, (1 << 19) - 20_000], 3, 50_000, 100),  # dense, alone only at the start and after a pull without compression
])
@pytest.mark.parametrize("flags", [0, dgs.DGS_RESIDUAL_MODE])
def test_one_kernel_and_two_in_turn(sizes, workers, ppm, join, flags):
    events = 6 * workers
    wl = W.custom("one", sizes, workers, events, ppm, grad_kind="normal")
    n, theta0 = sum(sizes), wl.theta0()
    orc = oracle.Oracle.from_workload(wl, theta0=theta0, residual_mode=bool(flags))
    ctx = dgs.Context.from_workload(wl, theta0=torch.from_numpy(theta0).to(DEV), flags=flags, pull_all_capacity=n)
    rng = np.random.default_rng(n)
    grads = [rng.standard_normal(n, dtype=np.float32) for _ in range(5)]
    on_gpu = [torch.from_numpy(g).to(DEV) for g in grads]
    torch.cuda.synchronize()
    for e in range(events):
        w, g = e % workers, e % 5
        if e % 9 == 5:                                # a pull without secondary compression on the same scratch
            push = ctx.worker_push(w, on_gpu[g])
            ctx.server_apply(w, push)
            gi, gv = ctx.var_packet(ctx.worker_pull_all(w))
            oi, ov = orc.push(w, grads[g])
            orc.apply(w, oi, ov)
            qi, qv, _ = orc.pull_all(w, n)
            assert np.array_equal(gi.cpu().numpy().view(np.uint32), qi) and np.array_equal(bits(gv.cpu().numpy()), bits(qv))
            continue
        got = ctx.event(w, on_gpu[g])
        want = orc.event(w, grads[g])
        if e % join == join - 1 or e == events - 1:
            for p, ref in zip(got, want):
                gi, gv = packet_to_numpy(ctx, p)
                assert np.array_equal(gi, ref[0]) and np.array_equal(bits(gv), bits(ref[1])), e
    assert ctx.status() == 0
    compare_state(ctx, orc, workers, False)


def test_a_pass_that_cannot_end_goes_no_further():
    """With DGS_TEST_STALLED_BARRIER the barrier between a pull's pass and its finalize waits for a CTA that does not exist, and
    the copies of the last CTA of a push's pass for an arrival that never comes: that CTA must leave at once, since finalize's
    tables lie where its copies land, and the others give up at the barrier.  Nothing after it may run."""
    n, k, workers = 300_000, 300, 3
    theta0 = torch.randn(n, device=DEV)
    ctx = dgs.Context(n, workers, 0.1, 0.9, [0], [n], [k], [k], theta0, flags=dgs.DGS_TEST_STALLED_BARRIER)
    grad = torch.randn(n, device=DEV)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for turn in range(6):                             # (the pairs of sync words are taken in turn)
        at = ctx.launch_count()
        ctx.worker_pull(turn % workers)               # alone; nothing to go by: two kernels for its bound, then one
        assert ctx.launch_count() == at + 3
        ctx.worker_push(turn % workers, grad)         # beside the pull
        assert ctx.launch_count() == at + (4 if turn else 6)   # the first push has nothing to go by either
        assert ctx.status() == dgs.DGS_ETIMEOUT
    assert time.perf_counter() - t0 < 20.0
    assert ctx.stats()[3] == 0                        # no finalize has looked at a candidate
    assert torch.equal(ctx.state(dgs.DGS_THETA), theta0)
    for w in range(workers):
        assert not ctx.state(dgs.DGS_U, w).any() and not ctx.state(dgs.DGS_D, w).any()
    ctx.close()
    test_one_kernel_and_two_in_turn([n], workers, 1_000, 3, 0)   # a context made afterwards runs clean


def launch_counter(sizes, workers):
    """A context that keeps a hundredth of every layer, and an event that returns how many kernels its push was."""
    n, ks = sum(sizes), [max(1, x // 100) for x in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    ctx = dgs.Context(n, workers, 0.1, 0.9, off, sizes, ks, ks, torch.zeros(n, device=DEV))
    grads = [torch.randn(n, device=DEV) for _ in range(workers)]

    def event(w):
        before = ctx.launch_count()
        pkt = ctx.worker_push(w, grads[w])
        launches = ctx.launch_count() - before
        ctx.server_apply(w, pkt)
        ctx.worker_pull(w)
        return launches
    return ctx, event


def test_an_event_that_opens_a_round_is_not_alone():
    """Alone on the GPU a push of a short vector is two kernels, beside other events one.  The event after a join is taken to be
    alone if the one before the join was, and to open a round if a round was before the join."""
    ctx, event = launch_counter([300_000], 3)
    for _ in range(2):
        for w in range(3):
            event(w)
        ctx.flush()
    assert [event(w) for w in range(3)] == [1, 1, 1]
    ctx.flush()
    event(0)
    ctx.flush()
    ctx.flush()                                   # a join with nothing before it says nothing
    assert event(1) == 2
    assert ctx.status() == 0
    assert [event(w) for w in range(3)] == [2, 1, 1]


@pytest.mark.parametrize("sizes,kernels", [
    ([LONGEST], 1),
    ([LONGEST + 1], 2),
    ([1 << 19, (1 << 19) - (2 << 13)], 1),            # two layers: 2^20 elements but 2^13 for each
    ([1 << 19, (1 << 19) - (2 << 13) + 1], 2),
    ([8_192] * 64, 1),                                # 2^19 from 64 layers on
    ([8_192] * 63 + [8_193], 2),
    ([64] * 512, 1),
    ([64] * 513, 2),
])
def test_which_selections_beside_other_events_are_one_kernel(sizes, kernels):
    ctx, event = launch_counter(sizes, 3)
    for _ in range(2):
        for w in range(3):
            event(w)
    assert [event(w) for w in range(3)] == [kernels] * 3
    assert ctx.status() == 0


@pytest.mark.parametrize("sizes", [[300_000], [100_000, 700, 50_000]])
@pytest.mark.parametrize("flags", [0, dgs.DGS_RESIDUAL_MODE])
def test_a_guess_that_fails_starts_over_inside_the_kernel(sizes, flags):
    """Every second round all values are a thousandth of what the carried bounds were made for, and no candidate is found."""
    workers, n = 3, sum(sizes)
    wl = W.custom("redo", sizes, workers, 1, 10_000, grad_kind="normal")
    orc = oracle.Oracle.from_workload(wl, residual_mode=bool(flags))
    ctx = dgs.Context.from_workload(wl, flags=flags)
    rng = np.random.default_rng(n)
    nothing = torch.zeros(n, device=DEV)
    for turn in range(6):
        scale = np.float32(1e-3 if turn % 2 else 1.0)
        grads = [rng.standard_normal(n, dtype=np.float32) * scale for _ in range(workers)]
        on_gpu = [torch.from_numpy(g).to(DEV) for g in grads]
        if turn % 2:
            for w in range(workers):
                for mine, its in ((dgs.DGS_U, oracle.U), (dgs.DGS_D, oracle.D)):
                    ctx.state_load(mine, w, nothing)
                    ctypes.memset(orc.state(its, w).ctypes.data, 0, 4 * n)
        torch.cuda.synchronize()
        before, launches = ctx.stats(), ctx.launch_count()
        for w in range(workers):
            got = ctx.event(w, on_gpu[w])
            want = orc.event(w, grads[w])
        if turn > 1:
            assert ctx.launch_count() - launches == 3 * workers      # push, apply, pull: a kernel each
        if turn % 2:
            assert ctx.stats()[1] > before[1]
        for p, ref in zip(got, want):
            gi, gv = packet_to_numpy(ctx, p)
            assert np.array_equal(gi, ref[0]) and np.array_equal(bits(gv), bits(ref[1])), turn
        compare_state(ctx, orc, workers, False)
    assert ctx.status() == 0
