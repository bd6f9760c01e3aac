"""The device step of small lattices (one TC row per lane) against the oracle's
replay: lattices held by one block and stepped by overlapping launches; sub-tiles that share a warp or fill it, with one and several band
columns, and a ragged last warp; draws on both, one or no rate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


SHAPES = [(64, 32, 16), (128, 64, 64), (192, 32, 32), (256, 64, 64), (384, 64, 16), (448, 32, 16),  # one block
          (576, 32, 32), (640, 64, 64), (1024, 32, 128), (1024, 128, 32),                           # launches of one-warp blocks
          (1088, 32, 16), (1152, 64, 64), (1088, 32, 32), (1280, 64, 32)]


@pytest.mark.parametrize("p,q", [(0.95, 0.05), (1.0, 0.0), (0.6, 0.0), (1.0, 0.5), (1.0, 1.0)])
@pytest.mark.parametrize("L,Bx,By", SHAPES)
def test_small_lattices_equal_oracle(g, oracle, L, Bx, By, p, q):
    prm = oracle.Params(L=L, p=p, q=q, seed=L + 3 * By, Bx=Bx, By=By)
    X, Y = oracle.flat(L)
    net, t = 0, 0
    with g.Simulation(L, p, q, L + 3 * By, Bx=Bx, By=By) as sim:
        for n in (1, 3):
            net += oracle.dtrdt_run(X, Y, prm, t, n)[0]
            sim.run(n)
            t += n
            Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
            assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
            m = sim.measure()
            assert (m.t, m.net_flips) == (t, net)


def test_long_run_of_a_small_lattice(g, oracle):
    """More MCS in one call than one launch takes."""
    L, n = 64, 1100
    prm = oracle.Params(L=L, p=0.95, q=0.05, seed=3, Bx=32, By=16)
    X, Y = oracle.flat(L)
    net = oracle.dtrdt_run(X, Y, prm, 0, n)[0]
    with g.Simulation(L, 0.95, 0.05, 3) as sim:
        sim.run(n)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
        assert sim.measure().net_flips == net


@pytest.mark.parametrize("L,Bx,By,scheme", [(256, 64, 64, 0), (1024, 64, 64, 0), (2048, 64, 64, 0), (1024, 256, 64, 0),
                                            (512, 64, 64, 1), (512, 64, 64, 2)])
def test_captured_run_replays(g, L, Bx, By, scheme):
    """oct_run_mcs captured into a CUDA graph: every replay advances the lattice
    by the captured MCS, with the counter that the kernels read."""
    import torch
    s = torch.cuda.Stream()
    with g.Simulation(L, 0.95, 0.05, 9, Bx=Bx, By=By, scheme=scheme) as ref:
        ref.run(1 + 2 * 3)
        want = ref.planes()
    with g.Simulation(L, 0.95, 0.05, 9, Bx=Bx, By=By, scheme=scheme, stream=s) as sim:
        sim.run(1)  # outside the graph: first-use set-up
        sim.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            sim.run(2)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(sim.planes(), want)


def test_device_steps_equal_a_run(g):
    from paper_1705_01022_gb300 import _lib
    L = 640
    with g.Simulation(L, 0.95, 0.05, 4) as a, g.Simulation(L, 0.95, 0.05, 4) as b:
        a.run(3)
        for _ in range(3):
            for k in range(4):
                _lib.oct_device_step(b.h, k)
            _lib.oct_end_mcs(b.h)
        assert np.array_equal(a.planes(), b.planes())
        assert a.measure().net_flips == b.measure().net_flips


def test_threads_with_different_sizes(g):
    """Threads on streams of their own, whose sizes and cells need different
    shared memory of the same kernels, get what each gets alone."""
    import threading

    import torch
    cases = [(64, 4, 4), (256, 4, 4), (512, 4, 4), (128, 8, 8), (512, 8, 8), (1024, 8, 8)]

    def once(L, cx, cy):
        with g.Simulation(L, 0.95, 0.05, L, cx=cx, cy=cy, stream=torch.cuda.Stream()) as sim:
            for _ in range(4):
                sim.run(1)
            return np.array(sim.lattice())

    want = [once(*c) for c in cases]
    bad = []

    def loop(i):
        try:
            for _ in range(10):
                if not np.array_equal(once(*cases[i]), want[i]):
                    bad.append(cases[i])
        except Exception as e:
            bad.append((cases[i], e))

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(cases))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not bad
