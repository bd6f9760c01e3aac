"""More jobs due at one tick than a batch keeps tickets for, and more results out
across ticks: every delivered W^2 equals the synchronous measurement of the same
replicas."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,times", [(1300, [1, 2, 4]), (300, [1, 2, 3, 4, 5, 6, 7, 8])], ids=["one tick", "across ticks"])
def test_every_result_is_delivered(n, times):
    import paper_1705_01022_gb300 as g
    from paper_1705_01022_gb300 import _lib, serve
    g.build()
    jobs = [serve.Job(i, 128 if i % 50 == 0 else 64, *serve.PQ_SET[i % 3], _lib.oct_replica_seed(4, i), times[-1],
                      measure_at=times) for i in range(n)]
    eng = serve.ServingEngine(1 << 30, max_inflight=8)
    try:
        done = eng.run(jobs)
        assert len(done) == n and not eng.pending
    finally:
        eng.close()
    with g.Batch([(j.L, j.p, j.q, j.seed, *j.shape) for j in jobs]) as b:
        t = 0
        for k, at in enumerate(times):
            b.run(at - t)
            t = at
            for j, m in zip(jobs, b.measure()):
                assert j.results[k] == (m.t, m.s1, m.s2, m.w2, m.net_flips), (j.jid, at)


def test_a_list_past_the_ring_is_refused():
    import paper_1705_01022_gb300 as g
    from paper_1705_01022_gb300 import _lib, serve
    g.build()
    b = serve.GpuBatch()
    try:
        slot = b.add(serve.Job(0, 64, 1.0, 0.0, 1, 1))
        assert len(b.measure_async_many([slot] * b.measure_limit)) == b.measure_limit
        with pytest.raises(_lib.OctError):
            b.measure_async_many([slot] * (b.measure_limit + 1))
    finally:
        b.close()
