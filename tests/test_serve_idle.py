"""Host logic of a solved group that its worker keeps open (`serve.py`): the bytes accounted for a request that
joins it, what its result and the batch's record say, and that nothing waits for it (fake backend)."""
import time

from test_serve import FakeBackend, expected, req, scat

import numpy as np

from paper_2111_11058_gb300 import serve as S


def _idle(srv, key, timeout=5.0):
    """Wait until the group of `key` is kept open after its solve."""
    end = time.perf_counter() + timeout
    while time.perf_counter() < end:
        with srv.lock:
            g = srv.open.get(key)
            if g is not None and g.state == "idle":
                return g
        time.sleep(0.0005)
    raise AssertionError("no idle group")


def _until(cond, timeout=5.0):
    end = time.perf_counter() + timeout
    while not cond() and time.perf_counter() < end:
        time.sleep(0.0005)
    assert cond()


def test_join_of_an_idle_group_is_accounted_in_full(monkeypatch):
    monkeypatch.setattr(S, "KEEP_OPEN_S", 5.0)
    sc = scat("a")
    be = FakeBackend(build_s=1.0, solve_s=0.2)     # a group stays open as long as its batch took
    srv = S.Server(be, hbm_budget=10**12, n_streams=1)
    n = S.estimate_n(sc, be.s)
    srv.submit(req(sc, 1.0, 4, 0)).result(timeout=30)
    _idle(srv, ("a", 1.0))
    assert srv.inflight == 0                                       # the session of the first solve is gone
    f = srv.submit(req(sc, 1.0, 6, 1))
    g = srv.open[("a", 1.0)]
    _until(lambda: g.state == "running")
    assert srv.inflight == S.solve_bytes(n, 6, sc.ne)
    f2 = srv.submit(req(sc, 1.0, 3, 2))                            # and one that joins the running session
    assert srv.inflight == S.solve_bytes(n, 9, sc.ne)
    for k, (x, nr) in enumerate(((f, 6), (f2, 3)), start=1):
        np.testing.assert_array_equal(x.result(timeout=30).rcs, expected(("a", 1.0), req(sc, 1.0, nr, k).exc))
    srv.drain(timeout=10)
    assert srv.inflight == 0
    srv.close()


def test_nothing_waits_for_an_idle_group(monkeypatch):
    monkeypatch.setattr(S, "KEEP_OPEN_S", 60.0)
    be = FakeBackend(build_s=1.5, solve_s=0.01)
    srv = S.Server(be, hbm_budget=10**12, n_streams=1)
    srv.submit(req(scat("a"), 1.0, 4, 0)).result(timeout=30)
    _idle(srv, ("a", 1.0))
    t0 = time.perf_counter()
    be.build_s = 0.01
    srv.submit(req(scat("b"), 1.0, 4, 1)).result(timeout=30)      # another key's request takes the worker
    assert time.perf_counter() - t0 < 1.0
    be.build_s = 1.5
    srv.submit(req(scat("c"), 1.0, 4, 2)).result(timeout=30)
    _idle(srv, ("c", 1.0))
    t0 = time.perf_counter()
    srv.drain(timeout=30)
    srv.close()
    assert time.perf_counter() - t0 < 1.0
    assert not any(srv.busy) and srv.inflight == 0


def test_a_request_on_the_resident_entry_is_a_hit(monkeypatch):
    """The batch that built the entry missed; a request solved later on the entry it left did not."""
    monkeypatch.setattr(S, "KEEP_OPEN_S", 5.0)
    sc = scat("a")
    srv = S.Server(FakeBackend(build_s=1.0, solve_s=0.01), hbm_budget=10**12, n_streams=1)
    first = srv.submit(req(sc, 1.0, 4, 0)).result(timeout=30)
    _idle(srv, ("a", 1.0))
    second = srv.submit(req(sc, 1.0, 4, 1)).result(timeout=30)
    srv.close()
    assert not first.cache_hit and second.cache_hit and second.batch_id == first.batch_id


class TimedBackend(FakeBackend):
    def event(self, st):
        return time.perf_counter()

    def elapsed_ms(self, e0, e1):
        return 1e3 * (e1 - e0)


def test_the_idle_gap_is_not_device_time(monkeypatch):
    monkeypatch.setattr(S, "KEEP_OPEN_S", 5.0)
    sc = scat("a")
    srv = S.Server(TimedBackend(build_s=1.0, solve_s=0.02), hbm_budget=10**12, n_streams=1)
    res = [srv.submit(req(sc, 1.0, 4, 0)).result(timeout=30)]
    _idle(srv, ("a", 1.0))
    time.sleep(0.2)
    res.append(srv.submit(req(sc, 1.0, 4, 1)).result(timeout=30))
    srv.drain(timeout=10)
    srv.close()
    assert len(srv.log) == 1 and srv.log[0]["requests"] == 2 and srv.log[0]["joined"] == 1
    a, b = srv.log[0]["dev_ms"]
    (c, d), = srv.log[0]["dev_later_ms"]
    assert b - a >= 1000 and c - b >= 190 and d - c >= 20
    stats = S.summarize(res, srv.log, 1.0, srv)
    assert abs(stats["device_busy_ms"] - (b - a) - (d - c)) < 1e-9
    assert stats["device_busy_ms"] < d - a - 190
