"""The serving loop around the library's server (no GPU): a server on a clock of its
own stands in for the library's."""
import pytest

from paper_0910_0329_gb300 import dpm, serve
from paper_0910_0329_gb300 import workloads as W

ROUND, POLL = 10.0, 1.0  # a round's time and that of one look at it


class FakeServer:
    """Rounds of fixed length; a request is done after two of them."""

    def __init__(self, slots):
        self.slots, self.t, self.state, self.left, self.flying, self.polls = slots, 0.0, {}, {}, [], 0
        self.n_rounds = self.max_active = 0

    def submit(self, geometry, source, seed):
        rid = len(self.state)
        self.state[rid], self.left[rid] = dpm.REQ_PENDING, 2
        return rid

    def active(self):
        return [r for r, s in self.state.items() if s == dpm.REQ_ACTIVE]

    def admit(self):
        for r, s in self.state.items():
            if s == dpm.REQ_PENDING and len(self.active()) < self.slots:
                self.state[r] = dpm.REQ_ACTIVE
        self.max_active = max(self.max_active, len(self.active()))

    def round_begin(self):
        assert not self.flying
        self.admit()
        self.flying, self.end = self.active(), self.t + ROUND
        return len(self.flying)

    def round_ready(self):
        self.polls += 1
        self.t += POLL
        return self.t >= self.end

    def round_end(self):
        self.t = max(self.t, self.end) if self.flying else self.t
        self.n_rounds += bool(self.flying)
        for r in self.flying:
            self.left[r] -= 1
            if not self.left[r]:
                self.state[r] = dpm.REQ_DONE
        self.flying = []

    def status(self, rid):
        return {"state": self.state[rid], "slot": rid, "histories": 100, "rounds": 2 - self.left[rid],
                "rel_sigma": 0.01, "dose_max": 1.0}

    def release(self, rid):
        self.state[rid] = dpm.REQ_RELEASED

    def info(self):
        return {"n_rounds": self.n_rounds, "histories": 0, "gpu_ms": 0.0, "max_active": self.max_active,
                "n_pending": sum(s == dpm.REQ_PENDING for s in self.state.values()), "peak_slot_bytes": 0}


@pytest.fixture
def server(monkeypatch):
    s = serve.Server.__new__(serve.Server)
    s.srv, s.template, s.seed_base, s.keep, s.fixed, s.stats = FakeServer(2), [0], 0, False, 0, serve.ServeStats()

    def sleep(dt):
        s.srv.t += dt

    monkeypatch.setattr(serve.time, "sleep", sleep)
    return s


def requests(*arrivals):
    src = W.Source(W.PHOTON, W.SPEC_6MV, 6.0, (1.0, 1.0, 1.0))
    return [serve.Request(k, 0, src, t) for k, t in enumerate(arrivals)]


@pytest.mark.parametrize("arrivals", [(0.0,), (0.0, 3.5), (0.0, 3.5, 4.0, 15.2, 100.0), (5.0, 5.0, 5.0, 6.0)])
def test_no_request_is_admitted_before_it_arrives(server, arrivals):
    st = server.run(requests(*arrivals), clock=lambda: server.srv.t)
    assert len(st.completed) == len(arrivals)
    for r in st.completed:
        assert r.arrival <= r.admitted <= r.done
    # the second request comes while the first one's round is under way and a slot is free
    if len(arrivals) > 1 and arrivals[1] == 3.5:
        r = next(r for r in st.completed if r.rid == 1)
        assert r.admitted - r.arrival <= 2 * POLL


def test_an_error_during_a_round_leaves_none_in_flight(server):
    submit = server.srv.submit
    server.srv.submit = lambda g, source, seed: submit(g, source, seed) if seed != 1 else 1 / 0
    with pytest.raises(ZeroDivisionError):
        server.run(requests(0.0, 3.5), clock=lambda: server.srv.t)
    assert server.srv.n_rounds == 1
    server.srv.submit = submit
    t0 = server.srv.t
    st = server.run(requests(0.0), clock=lambda: server.srv.t - t0)
    assert len(st.completed) == 1
