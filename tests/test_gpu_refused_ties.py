"""Rates that are multiples of 1/16, whose tied uniforms are all refused, against
the oracle's replay: every block layer and cell on lane rows, packed and full
warps, the finest other rates beside them, and batches that mix both in a warp."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -32
RATES = [(0.5, 0.5), (0.0625, 0.9375), (0.25, 0.0), (1.0, 0.75), (0.5 + EPS, 0.5), (0.5, 0.25 - EPS)]
FORMS = [(128, 64, 64, 0, 4, 4), (192, 32, 32, 0, 4, 4), (192, 96, 16, 0, 4, 4), (256, 128, 64, 0, 4, 4),
         (512, 256, 64, 0, 4, 4), (256, 64, 64, 1, 4, 4), (512, 256, 64, 1, 4, 4), (256, 64, 64, 3, 4, 4),
         (512, 256, 64, 3, 4, 4), (256, 64, 64, 0, 8, 8), (512, 256, 64, 0, 8, 8), (256, 64, 64, 0, 16, 16),
         (512, 256, 64, 0, 16, 8), (128, 32, 32, 0, 8, 4)]


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


@pytest.mark.parametrize("p,q", RATES)
@pytest.mark.parametrize("L,Bx,By,scheme,cx,cy", FORMS)
def test_lattices_equal_oracle(g, oracle, L, Bx, By, scheme, cx, cy, p, q):
    prm = oracle.Params(L=L, p=p, q=q, seed=L + By, Bx=Bx, By=By, cx=cx, cy=cy, scheme=scheme)
    X, Y = oracle.flat(L)
    net = oracle.dtrdt_run(X, Y, prm, 0, 3)[0]
    with g.Simulation(L, p, q, L + By, Bx=Bx, By=By, cx=cx, cy=cy, scheme=2 if scheme == 3 else scheme) as sim:
        sim.run(3)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
        assert sim.measure().net_flips == net


@pytest.mark.parametrize("copies", [1, 24])
def test_batches_of_both_kinds_equal_single_runs(g, copies):
    """One copy runs in row lanes, many replicas (with large ones) on packed warps."""
    reps = [(L, p, q, 7 + 5 * L + i) for i, (p, q) in enumerate(RATES + [(0.95, 0.05)]) for L in (64, 128)] * copies
    reps += [(4096, 0.5, 0.5, 3 + i) for i in range(9 if copies > 1 else 0)]
    with g.Batch(reps) as b:
        b.run(5)
        for r in list(range(14)) + list(range(14 * copies, len(reps))):
            L, p, q, seed = reps[r]
            with g.Simulation(L, p, q, seed, Bx=64 if L % 128 == 0 else 32, By=64 if L % 128 == 0 else 32) as sim:
                sim.run(5)
                assert np.array_equal(b.planes(r), sim.planes())
