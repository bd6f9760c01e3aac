"""Exact roughness of lattices up to 16384 sites a side (rows split over part
of a warp, one launch for many lattices): the sums equal the oracle's at the
edges of the split, and a batch's measurement equals its replicas' own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1705_01022_gb300 as g
    g.build()
    return g


# words per row 2 .. 512: rows sharing a warp, partly filled lanes (L = 320, 2112, 4160), one and
# several words per lane
@pytest.mark.parametrize("L", [64, 128, 192, 320, 1024, 1088, 2112, 4096, 4160, 8256])
def test_sums_equal_oracle(g, oracle, L):
    import torch
    rng = np.random.default_rng(L)
    X = rng.integers(0, 2, (L, L), dtype=np.uint8)
    Y = rng.integers(0, 2, (L, L), dtype=np.uint8)
    X[:3], Y[:, 0] = 1, 1  # monotone rows and a monotone column: the largest heights
    words = oracle.pack_planar(X, Y)
    lat = torch.from_numpy(words.view(np.int32).copy()).cuda()
    from paper_1705_01022_gb300 import _lib
    m = _lib.oct_w2_noalloc(lat.data_ptr(), L, None)
    h0 = np.concatenate([[0], np.cumsum(2 * Y[1:, 0].astype(np.int64) - 1)])
    h = np.cumsum(2 * X.astype(np.int64) - 1, axis=1)
    h += (h0 - h[:, 0])[:, None]
    assert (m.s1, m.s2, m.hmax) == (int(h.sum()), int((h * h).sum()), int(np.abs(h).max()))
    s1, s2, _ = oracle.w2_sums(X, Y)
    assert (m.s1, m.s2) == (s1, s2)


def test_batch_measure_equals_slots(g):
    from paper_1705_01022_gb300 import _lib
    reps = [(64 * (1 + (7 * i) % 33), *((1.0, 0.0), (0.9, 0.2))[i % 2], 100 + i) for i in range(37)]
    with g.Batch(reps) as b:
        b.run(3)
        for r in (0, 5, 36):
            _lib.oct_batch_remove(b.h, r)
        b.run(2)
        for again in range(2):
            for i, m in enumerate(b.measure()):
                if i in (0, 5, 36):
                    assert (m.n_sites, m.s1, m.s2, m.t) == (0, 0, 0, 0)
                    continue
                o = _lib.oct_batch_measure_slot(b.h, i)
                assert (m.t, m.s1, m.s2, m.hmax, m.net_flips, m.w2) == (5 + again, o.s1, o.s2, o.hmax, o.net_flips, o.w2)
            b.run(1)


def test_batch_measure_in_several_launches(g):
    """66 replicas of L = 16384 have more rows than one launch takes (2^20)."""
    L = 16384
    with g.Batch([(L, 1.0, 0.0, i, 256, 64) for i in range(66)]) as b:
        for m in b.measure():
            assert (m.s1, m.s2, m.hmax, m.w2) == (L * L // 2, L * L // 2, 1, 0.25)
