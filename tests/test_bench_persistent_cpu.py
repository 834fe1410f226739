"""bench.py's persistent leg reports the persistent form or nothing (no GPU)."""
import os

import bench


class FakeLibrary:
    """A library whose graphs hold `launches` kernels; running one is not expected."""
    MODE_DCF = 1

    def __init__(self, launches):
        self.launches, self.count, self.closed = launches, 99, 0

    def launch_count_reset(self):
        self.count = 0

    def launch_count(self):
        return self.count

    def Batch(self, plans, fs, hs, mode):
        assert os.environ["INFFT_PERSISTENT"] == "1"
        self.count += self.launches
        return self

    def run(self):
        raise AssertionError("timed the staged kernels")

    def close(self):
        self.closed += 1


class FakeTorch:
    @staticmethod
    def empty_like(h):
        return h


def test_staged_graph_is_not_reported_as_the_persistent_form(monkeypatch):
    monkeypatch.delenv("INFFT_PERSISTENT", raising=False)
    L = FakeLibrary(3)
    out = bench.persistent_leg(L, FakeTorch, [None], [None], [None], 5, None)
    assert set(out) == {"unavailable"} and "3 launches" in out["unavailable"]
    assert L.closed == 1 and "INFFT_PERSISTENT" not in os.environ
