"""A long run of a small batch: the call returns before the device is done, and
the lattices equal the plain runs, at every split into launches and replays."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

REPS = [(128, 0.95, 0.05, 3), (64, 1.0, 0.0, 4), (192, 0.5, 0.5, 5), (320, 0.6, 0.0, 6)]


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


def _check(g, b, t):
    ms = b.measure()
    for i, (L, p, q, seed) in enumerate(REPS):
        B = 64 if L % 128 == 0 else 32
        with g.Simulation(L, p, q, seed, Bx=B, By=B) as sim:
            sim.run(t)
            assert np.array_equal(b.planes(i), sim.planes()), (i, t)
            assert ms[i].t == t and ms[i].net_flips == sim.measure().net_flips


@pytest.mark.parametrize("runs", [(128, 8, 7, 9, 32, 31), (135, 1), (136, 160, 3), (400,), (8,) * 20, (100, 100, 100)])
def test_splits_equal_plain_runs(g, runs):
    with g.Batch(REPS) as b:
        for n in runs:
            b.run(n)
        _check(g, b, sum(runs))


def test_membership_change_after_replays(g):
    from paper_1705_01022_gb300 import _lib
    with g.Batch(REPS) as b:
        b.run(300)
        r = _lib.oct_replica()
        r.L, r.p, r.q, r.seed = 256, 0.9, 0.1, 77
        slot = _lib.oct_batch_add(b.h, r)
        b.run(200)
        _lib.oct_batch_remove(b.h, slot)
        b.run(37)
        ms = [_lib.oct_batch_measure_slot(b.h, i) for i in range(len(REPS))]
        for i, (L, p, q, seed) in enumerate(REPS):
            B = 64 if L % 128 == 0 else 32
            with g.Simulation(L, p, q, seed, Bx=B, By=B) as sim:
                sim.run(537)
                m = sim.measure()
                assert (ms[i].t, ms[i].s1, ms[i].net_flips) == (537, m.s1, m.net_flips)


def test_in_a_callers_capture(g):
    """A stream that is being captured takes the launches."""
    import torch
    s = torch.cuda.Stream()
    with g.Batch(REPS, stream=s) as b:
        b.run(130)
        b.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            b.run(40)
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        _check(g, b, 210)


def test_long_run_returns_before_the_device_is_done(g):
    """(Launch by launch, the call waits until about a thousand launches are left:
    9/10 of this run.)"""
    with g.Batch(REPS) as b:
        b.run(1)
        b.sync()
        t0 = time.perf_counter()
        b.run(3000)
        t1 = time.perf_counter()
        b.sync()
        t2 = time.perf_counter()
        print(f"call {1e3 * (t1 - t0):.2f} ms of {1e3 * (t2 - t0):.2f} ms")
        assert t1 - t0 < 0.5 * (t2 - t0)
