"""Served requests over more than 65,536 edges that do not get their memory while
small requests hold it wait for it, and are answered."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MB = 1 << 20


def _pairs(n, at=0):
    """n disjoint edges: the closure is the edges."""
    a = np.arange(n, dtype=np.uint32) + np.uint32(at)
    return a, a + np.uint32(n)


def _closed(src, dst):
    return np.unique(src.astype(np.uint64) << np.uint64(32) | dst.astype(np.uint64))


def _drain(c):
    while c.serve_step(16):
        pass


def test_first_buffers_beside_running_lanes():
    # small requests whose bit sets take 128 MB while they run; the large one asks
    # for 290 of 400 MB at its start
    from paper_2607_17571_gb300 import wg
    small = [_pairs(8000, 100_000 * k) for k in range(4)]
    i = np.arange(70_000, dtype=np.uint32)
    big = (i % 4500, np.uint32(5000) + (i // 4500 * 271 + i % 4500 * 7) % 4500)
    with wg.Context(0, mem_budget=400 * MB, torch_memory=False) as c:
        rels = [c.load(*e) for e in small + [big]]
        hs = c.submit([(wg.WG_TC, r) for r in rels[:4]] +
                      [(wg.WG_TC, rels[4], dict(reserve_full=290 * MB // 4))])
        _drain(c)
        for e, h in zip(small + [big], hs):
            h.wait()
            assert np.array_equal(h.result(), _closed(*e))
            h.free()
