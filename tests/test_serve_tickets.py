"""More measurements out than a batch keeps results for: the engine reads the
oldest before their tickets expire, and every job still gets all its results in
order (no GPU: a batch with a small ring of tickets)."""
import pytest

from paper_1705_01022_gb300 import serve


class RingBatch:
    """Results of the last `measure_limit` tickets; one is ready only after
    `lag` further runs (a device behind the host)."""

    def __init__(self, limit, lag, many):
        self.measure_limit, self.lag = limit, lag
        self.slots, self.t, self.runs, self.tickets, self.waits = {}, {}, 0, [], 0
        self.next = 0
        if many:
            self.measure_async_many = lambda slots: [self.measure_async(s) for s in self._checked(slots)]

    def _checked(self, slots):
        assert len(slots) <= self.measure_limit
        return slots

    def add(self, job):
        self.next += 1
        self.slots[self.next], self.t[self.next] = job, 0
        return self.next

    def remove(self, slot):
        del self.slots[slot]

    def run(self, n):
        self.runs += 1
        for s in self.slots:
            self.t[s] += n

    def measure_async(self, slot):
        self.tickets.append(((self.t[slot], self.slots[slot].jid, 0, 0.0, 0), self.runs))
        return len(self.tickets) - 1

    def _live(self, ticket):
        if ticket < len(self.tickets) - self.measure_limit:
            raise RuntimeError("expired measurement ticket")
        return self.tickets[ticket]

    def poll(self, ticket):
        res, at = self._live(ticket)
        return res if self.runs > at + self.lag else None

    def wait(self, ticket):
        self.waits += 1
        return self._live(ticket)[0]


@pytest.mark.parametrize("many", [True, False])
@pytest.mark.parametrize("n_batches", [1, 2])
@pytest.mark.parametrize("limit,jobs,lag", [(8, 40, 0), (8, 9, 5), (8, 3, 20), (1, 5, 2), (7, 7, 1)])
def test_no_ticket_expires(limit, jobs, lag, n_batches, many):
    batches = [RingBatch(limit, lag, many) for _ in range(n_batches)]
    seen = []
    eng = serve.ServingEngine(1 << 30, batch=batches, on_result=lambda j, r: seen.append((j.jid, r[0])))
    todo = [serve.Job(i, 64, 1.0, 0.0, i, t_max=9 + i % 2, measure_at=list(range(1, 10 + i % 2))) for i in range(jobs)]
    done = eng.run(todo)
    assert len(done) == jobs and not eng.pending and not any(eng.unread)
    for j in todo:
        assert [r[0] for r in j.results] == j.measure_at and all(r[1] == j.jid for r in j.results)
        assert [t for jid, t in seen if jid == j.jid] == j.measure_at
    assert len(seen) == sum(len(j.measure_at) for j in todo)


def test_ordinary_load_never_waits():
    b = RingBatch(64, 1, True)
    eng = serve.ServingEngine(1 << 30, batch=b)
    eng.run([serve.Job(i, 64, 1.0, 0.0, i, t_max=6, measure_at=[1, 2, 3, 4, 5, 6]) for i in range(16)])
    assert b.waits <= 16 * 2  # the last ticks' results, once nothing runs any more
