"""Rounds of a power iteration in the serving loop (CPU: the device side is replaced by a clock that every
launch advances): a request that arrives while rounds are being launched joins after the round at hand."""
import pytest

from paper_2308_00106_gb300 import serve


class _Stream:
    def wait_stream(self, other):
        pass


class _Done:
    def query(self):
        return True


class _Server(serve.Server):
    """The loop alone: every product takes one second of the host's clock and is done when it is launched."""

    def __init__(self, clock, streams):
        self.clock, self.log = clock, []
        self.capacity, self.step_bytes, self.backlog_bytes = 4096, 1 << 30, 1 << 32
        self.mem_cap, self.resident_bytes = 1 << 40, 0
        self.streams, self.adm_stream = [_Stream() for _ in range(streams)], _Stream()

    def request_bytes(self, r):
        return 1

    def unit_bytes(self, r):
        return 1

    def _admit(self, r, stream):
        pass

    def _launch(self, si, reqs):
        for r in reqs:
            self.log.append((self.clock[0], r.rid))
            r.units_done += 1
        self.clock[0] += 1.0

    def _event(self, si):
        return _Done()

    def _finish(self, r, keep):
        pass


@pytest.mark.parametrize("streams", [1, 2])
def test_an_arrival_joins_after_the_round_at_hand(monkeypatch, streams):
    clock = [0.0]
    monkeypatch.setattr(serve.time, "perf_counter", lambda: clock[0])
    monkeypatch.setattr(serve.time, "sleep", lambda s: clock.__setitem__(0, clock[0] + 1e-3))
    srv = _Server(clock, streams)
    power = serve.Request(0, 0.0, 0, "power", steps=100)
    late = [serve.Request(1 + i, 10.5 + 20 * i, 0, "spmv") for i in range(3)]
    stats = srv.run([power, *late])
    assert stats["requests"] == 4 and power.units_done == 101
    for r in late:  # launched within two rounds of its arrival, long before the power iteration ends
        at = next(t for t, rid in srv.log if rid == r.rid)
        assert r.arrival <= at <= r.arrival + 2.0, (r.rid, at)
        assert r.t_done < power.t_done


def test_rounds_still_share_a_step_when_nobody_arrives(monkeypatch):
    clock = [0.0]
    monkeypatch.setattr(serve.time, "perf_counter", lambda: clock[0])
    srv = _Server(clock, 2)
    power = serve.Request(0, 0.0, 0, "power", steps=100)
    stats = srv.run([power, serve.Request(1, 0.0, 0, "spmv")])
    assert stats["batch_steps"] <= 4
