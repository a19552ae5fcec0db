"""The batched and served passes of bench.py count all time from the first
submission to the last completion: other queries' launches run on while one is
checked, so nothing done in between may be taken off the clock."""
import os
import sys
import time
from types import SimpleNamespace

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


class _Ctx:
    """Queries that complete one per step; `check` below stands for a slow one."""

    def __init__(self):
        self.left, self.n = [], 0

    def submit(self, reqs):
        hs = []
        for _ in reqs:
            self.n += 1
            st = SimpleNamespace(error=0, state=2, n_tuples=7, iterations=1)
            hs.append(SimpleNamespace(id=self.n, poll=lambda st=st: st, free=lambda: None))
            self.left.append(self.n)
        return hs

    def serve_step(self, iters):
        return len(self.left)

    def take_completed(self):
        return [self.left.pop(0)] if self.left else []


def _slow(i, h, st):
    time.sleep(0.01)
    return int(i == 3)


def test_batched_pass_counts_the_checks():
    s, lat, tuples, bad = bench.batched_pass(_Ctx(), [None] * 8, 16, _slow)
    assert s >= 0.08 and tuples == 56 and bad == 1
    assert all(x >= 10 * i for i, x in enumerate(lat))


def test_served_pass_counts_the_checks():
    r = bench.served_pass(_Ctx(), [None] * 4, [0.0] * 8, 60.0, 16, _slow)
    assert r["seconds"] >= 0.08 and r["completed"] == 8 and r["parity_failures"] == 2
    assert r["queries_per_s"] <= 100 and r["unfinished_in_time"] == 0
