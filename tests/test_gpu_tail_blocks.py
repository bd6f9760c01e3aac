"""oct_stats.tail_blocks as the header states it: none without acceptance draws,
and none where both rates lie strictly inside (0, 1) and are multiples of 1/16, on
every block layer and form of the step; some with finer rates."""
import pytest

pytestmark = pytest.mark.gpu

FORMS = [(256, 64, 64, 0, 4, 4), (640, 64, 64, 0, 4, 4), (192, 32, 32, 0, 4, 4), (192, 96, 16, 0, 4, 4), (512, 256, 64, 0, 4, 4),
         (256, 64, 64, 1, 4, 4), (512, 256, 64, 1, 4, 4), (256, 64, 64, 2, 4, 4), (512, 256, 64, 2, 4, 4),
         (256, 64, 64, 0, 16, 16), (512, 256, 64, 0, 8, 8), (128, 32, 32, 0, 4, 8)]


@pytest.mark.parametrize("p,q,some", [(0.5, 0.5, False), (0.0625, 0.9375, False), (0.75, 0.125, False), (1.0, 0.0, False),
                                      (1.0, 1.0, False), (0.95, 0.05, True)])
@pytest.mark.parametrize("L,Bx,By,scheme,cx,cy", FORMS)
def test_tail_blocks(L, Bx, By, scheme, cx, cy, p, q, some):
    import paper_1705_01022_gb300 as g
    from paper_1705_01022_gb300 import _lib
    g.build()
    with g.Simulation(L, p, q, 5, Bx=Bx, By=By, cx=cx, cy=cy, scheme=scheme) as sim:
        sim.run(3)
        assert (_lib.oct_get_stats(sim.h).tail_blocks > 0) == some
