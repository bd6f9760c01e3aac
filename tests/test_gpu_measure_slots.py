"""Asynchronous W^2 of several replicas in one call equals the synchronous one
of each: lists longer than one launch takes, by count and by rows, a slot named
twice, tickets past the end of their ring, a removal right after the call."""
import pytest

pytestmark = pytest.mark.gpu

FIELDS = ("t", "s1", "s2_lo", "s2_hi", "hmax", "net_flips", "w2")


def _values(m):
    return tuple(getattr(m, f) for f in FIELDS)


@pytest.mark.parametrize("sizes", [[64], [64, 128] * 17, [4096] * 17 + [64] * 3, [64, 192, 512, 96 * 2, 2048]],
                         ids=["one", "count", "rows", "mixed"])
def test_lists_equal_single_measurements(sizes):
    import paper_1705_01022_gb300 as g
    from paper_1705_01022_gb300 import _lib
    g.build()
    with g.Batch([(L, 0.95, 0.05, 31 + i) for i, L in enumerate(sizes)]) as b:
        slots = list(range(len(sizes))) + [0]
        for rnd in range(2):
            b.run(1 + rnd)
            for _ in range(1 + 1100 * rnd // len(slots)):  # the second round passes the ring's end
                tickets = _lib.oct_batch_measure_slots_async(b.h, slots)
            want = [_values(_lib.oct_batch_measure_slot(b.h, s)) for s in slots]
            assert [_values(_lib.oct_batch_wait(b.h, t)) for t in tickets] == want
            assert [_values(_lib.oct_batch_poll(b.h, t)) for t in tickets] == want
        b.run(1)
        tickets = _lib.oct_batch_measure_slots_async(b.h, slots)
        want = [_values(_lib.oct_batch_measure_slot(b.h, s)) for s in slots]
        tickets += _lib.oct_batch_measure_slots_async(b.h, slots[-1:])
        _lib.oct_batch_remove(b.h, 0)
        assert [_values(_lib.oct_batch_wait(b.h, t)) for t in tickets] == want + want[-1:]
        before = tickets[-1]
        for bad in ([0], [1, 0], [len(sizes) + 5], [-1]):  # nothing is enqueued when one slot is refused
            with pytest.raises(_lib.OctError):
                _lib.oct_batch_measure_slots_async(b.h, bad)
        with pytest.raises(_lib.OctError):
            _lib.oct_batch_wait(b.h, before + 1)
        assert _lib.oct_batch_measure_slots_async(b.h, []) == []


@pytest.mark.parametrize("L", [8192, 8256])
def test_one_large_replica(L):
    """The last size one block finishes and the first it does not: alone, listed
    with another, and as a simulation."""
    import paper_1705_01022_gb300 as g
    from paper_1705_01022_gb300 import _lib
    g.build()
    with g.Simulation(L, 0.95, 0.05, 5, Bx=32, By=32) as sim:
        sim.run(2)
        m = sim.measure()
        want = tuple(getattr(m, f) for f in FIELDS)
    rep = (L, 0.95, 0.05, 5, 32, 32)
    with g.Batch([rep]) as b, g.Batch([rep, rep]) as two:
        for x in (b, two):
            x.run(2)
        got = [_values(m) for m in b.measure() + two.measure()]
        got += [_values(_lib.oct_batch_measure_slot(b.h, 0))]
        got += [_values(_lib.oct_batch_wait(x.h, t)) for x in (b, two)
                for t in _lib.oct_batch_measure_slots_async(x.h, list(range(len(x))))]
    assert got == [want] * 7
