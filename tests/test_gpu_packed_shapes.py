"""Several sub-tiles in one warp, for every block layer: lattice and net flips
equal the oracle's for power-of-two and other group counts (a sub-tile of six
groups leaves two lanes of its eight without a group), with one, several and
a ragged last warp of sub-tiles, and for draws on both, one or no rate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


@pytest.mark.parametrize("scheme", ["dt", "db", "dtr"])
@pytest.mark.parametrize("p,q", [(0.95, 0.05), (1.0, 0.0), (0.7, 0.0), (1.0, 1.0)])
@pytest.mark.parametrize("L,Bx,By", [(64, 32, 16), (192, 32, 32), (192, 96, 32), (384, 96, 16), (384, 64, 48),
                                     (640, 64, 64), (512, 128, 32), (512, 32, 256)])
def test_packed_subtiles_equal_oracle(g, oracle, scheme, L, Bx, By, p, q):
    n = 4
    prm = oracle.Params(L=L, p=p, q=q, seed=L + By, Bx=Bx, By=By, scheme={"dt": 0, "db": 1, "dtr": 3}[scheme])
    X, Y = oracle.flat(L)
    net = oracle.dtrdt_run(X, Y, prm, 0, n)[0]
    with g.Simulation(L, p, q, L + By, Bx=Bx, By=By, scheme={"dt": 0, "db": 1, "dtr": 2}[scheme]) as sim:
        sim.run(n)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
        assert sim.measure().net_flips == net
