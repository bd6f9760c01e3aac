"""A batch small enough for row lanes (one launch per device step for all modes)
equals its plain runs, also when it grows past that size and shrinks again, and
when its sub-tiles do not allow it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RATES = [(1.0, 0.0), (0.95, 0.05), (0.6, 0.0), (0.0, 1.0), (1.0, 1.0), (1.0, 0.5), (0.0, 0.0)]


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


def _same(g, b, i, r, t):
    L, p, q, seed = r[:4]
    Bx, By = r[4:] if len(r) > 4 else ((64, 64) if L % 128 == 0 else (32, 32))
    with g.Simulation(L, p, q, seed, Bx=Bx, By=By) as sim:
        sim.run(t)
        assert np.array_equal(b.planes(i), sim.planes()), (i, r)
        return sim.measure()


def test_rows_equal_plain_runs(g):
    shapes = [(64,), (128,), (192,), (320,), (256, 32, 16), (256, 128, 32), (512, 32, 128), (384, 64, 32)]
    reps = [(s[0], *RATES[(i + j) % len(RATES)], 50 + 10 * i + j, *s[1:])
            for i, s in enumerate(shapes) for j in range(len(RATES))]
    with g.Batch(reps) as b:
        for n in (1, 4, 3):
            b.run(n)
        ms = b.measure()
        for i, r in enumerate(reps):
            m = _same(g, b, i, r, 8)
            assert (ms[i].t, ms[i].s1, ms[i].s2, ms[i].net_flips) == (8, m.s1, m.s2, m.net_flips)


def test_membership_moves_between_rows_and_graphs(g):
    from paper_1705_01022_gb300 import _lib
    small = [(128 * (1 + i % 4), *RATES[i % 3], 7 + i) for i in range(9)]

    def replica(L, p, q, seed, Bx=0, By=0):
        r = _lib.oct_replica()
        r.L, r.p, r.q, r.seed, r.Bx, r.By = L, p, q, seed, Bx, By
        return r

    with g.Batch(small) as b:
        b.run(5)
        wide = _lib.oct_batch_add(b.h, replica(512, 0.9, 0.1, 99, 256, 64))   # a full-warp sub-tile
        b.run(6)
        assert _lib.oct_batch_measure_slot(b.h, wide).t == 6
        _lib.oct_batch_remove(b.h, wide)
        big = [_lib.oct_batch_add(b.h, replica(8192, 1.0, 0.0, 5 + i)) for i in range(2)]  # 134 M sites
        b.run(5)
        for s in big:
            _lib.oct_batch_remove(b.h, s)
        b.run(2)
        for i, r in enumerate(small):
            _same(g, b, i, r, 18)
            assert _lib.oct_batch_measure_slot(b.h, i).t == 18
