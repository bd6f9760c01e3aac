"""The row-lane device step in blocks of four warps, and the sizes on both sides
of the lines between one-warp blocks, four-warp blocks and packed groups, against
the oracle's replay of one MCS: a sub-tile per warp and four to a warp, ragged last
blocks and warps, every acceptance mode."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KPZ, TIES, EW, ONE = (1.0, 0.0), (0.95, 0.05), (0.5, 0.5), (0.6, 0.0)
# warps of a device step: 3041..4864 take blocks of four, fewer one-warp blocks, more packed groups
CASES = [(7040, 64, TIES),                                                  # 3025: the last in one-warp blocks
         (7168, 64, KPZ), (7168, 64, TIES), (7168, 64, EW), (7168, 64, ONE),  # 3136
         (7296, 64, EW),                                                    # 3249: one warp in the last block
         (8832, 64, KPZ), (8832, 64, TIES),                                 # 4761
         (8960, 64, TIES),                                                  # 4900: the first in packed groups
         (7040, 32, EW),                                                    # 3025, four sub-tiles to a warp
         (7104, 32, KPZ), (7104, 32, TIES), (7104, 32, EW), (7104, 32, ONE),  # 3081, the last warp with one sub-tile
         (8896, 32, TIES), (8896, 32, EW),                                  # 4831
         (8960, 32, KPZ)]                                                   # 4900


@pytest.fixture(scope="module")
def replays(oracle):
    """The oracle's lattices (bits packed) and net flips, all cases at once: its C
    code runs outside the interpreter's lock."""
    def one(case):
        L, B, (p, q) = case
        X, Y = oracle.flat(L)
        net = oracle.dtrdt_run(X, Y, oracle.Params(L=L, p=p, q=q, seed=L + B, Bx=B, By=B), 0, 1)[0]
        return np.packbits(X), np.packbits(Y), net

    with ThreadPoolExecutor(8) as ex:
        return dict(zip(CASES, ex.map(one, CASES)))


@pytest.mark.parametrize("case", CASES, ids=str)
def test_one_mcs_equals_oracle(oracle, replays, case):
    import paper_1705_01022_gb300 as g
    g.build()
    L, B, (p, q) = case
    X, Y, net = replays[case]
    with g.Simulation(L, p, q, L + B, Bx=B, By=B) as sim:
        sim.run(1)
        Xg, Yg = oracle.unpack_canonical(sim.lattice(), L)
        assert np.array_equal(np.packbits(Xg), X) and np.array_equal(np.packbits(Yg), Y)
        assert sim.measure().net_flips == net
