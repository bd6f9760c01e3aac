"""Coarse thread cells with one lane per cell against the oracle's replay: cells
of every width and height the kernel has, sub-tiles that fill part of a warp
(several share it), a warp and several turns of one, incomplete group rows
(fewer than four rows of cells), band columns that are no power of two, and
draws on both, one or no rate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


CELLS = [(8, 4), (16, 4), (32, 4), (8, 8), (16, 8), (32, 8), (8, 16), (16, 16), (32, 16)]
SHAPES = [(64, 32, 16), (192, 32, 32), (192, 96, 48), (256, 64, 64), (256, 32, 128), (512, 256, 64), (320, 32, 80)]


@pytest.mark.parametrize("p,q", [(0.95, 0.05), (1.0, 0.0), (0.6, 0.0), (1.0, 0.5), (1.0, 1.0)])
@pytest.mark.parametrize("L,Bx,By", SHAPES)
@pytest.mark.parametrize("cx,cy", CELLS)
def test_lane_cells_equal_oracle(g, oracle, L, Bx, By, cx, cy, p, q):
    n = 2
    prm = oracle.Params(L=L, p=p, q=q, seed=L + 7 * cx + cy, Bx=Bx, By=By, cx=cx, cy=cy)
    X, Y = oracle.flat(L)
    net = oracle.dtrdt_run(X, Y, prm, 0, n)[0]
    with g.Simulation(L, p, q, L + 7 * cx + cy, Bx=Bx, By=By, cx=cx, cy=cy) as sim:
        sim.run(n)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(Xg, X) and np.array_equal(Yg, Y)
        assert sim.measure().net_flips == net
