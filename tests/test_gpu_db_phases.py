"""DTrDB with both rates non-zero (bulk, border and corner attempts of a step
decided in turn) against the oracle's replay, at the shapes where a border
attempt's neighbour cell is in the same lane, the next lane, the next lane
row or outside the sub-tile, and for draws on both, one or neither rate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


@pytest.mark.parametrize("p,q", [(0.95, 0.05), (0.5, 0.5), (1.0, 0.5), (0.4, 1.0), (1.0, 1.0)])
@pytest.mark.parametrize("L,Bx,By", [(128, 32, 16), (256, 64, 64), (256, 128, 16), (256, 32, 128), (512, 256, 64),
                                     (1024, 512, 32), (1024, 32, 512), (2048, 1024, 16)])
def test_delayed_borders_equal_oracle(g, oracle, L, Bx, By, p, q):
    prm = oracle.Params(L=L, p=p, q=q, seed=L + Bx, Bx=Bx, By=By, scheme=1)
    X, Y = oracle.flat(L)
    net = oracle.dtrdt_run(X, Y, prm, 0, 3)[0]
    with g.Simulation(L, p, q, L + Bx, Bx=Bx, By=By, scheme=1) as sim:
        sim.run(3)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
        assert sim.measure().net_flips == net
