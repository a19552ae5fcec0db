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


def _long_rows(rows):
    """`rows` rows of 261 tuples over 400,000 vertices."""
    i, hubs = np.arange(rows), np.arange(30_000, 30_010)
    src = np.concatenate([np.arange(0, 400_000, 2), i, np.repeat(hubs, 260)]).astype(np.uint32)
    dst = np.concatenate([np.arange(1, 400_001, 2), 30_000 + i % 10,
                          np.tile(np.arange(50_000, 50_260), 10)]).astype(np.uint32)
    return src, dst


@pytest.mark.parametrize("budget_mb,reserve_mb", [
    (2600, 900),   # rows never fit (1.8 GB beside the reserve); the pipeline's start waits
    (2600, 300),   # rows fit once the engine of the small request is gone
    (2600, 20),    # ... with less to reserve
    (2000, 20)])   # the relation's lists are over half of what is free: the pipeline
def test_long_rows_beside_a_batch_engine(budget_mb, reserve_mb):
    # a submitted query that asks for candidate buffers has a batch engine, whose
    # pools take a third of the budget; bit sets of the large one's rows 1.4 GB
    from oracle import oracle_tc_reach
    from paper_2607_17571_gb300 import wg
    src, dst = _long_rows(26_000)
    n, iters, log, dg = oracle_tc_reach(src, dst, n_threads=8)
    small = _pairs(5000)
    with wg.Context(0, mem_budget=budget_mb * MB, torch_memory=False) as c:
        a, b = c.load(*small), c.load(src, dst)
        hs = c.submit([(wg.WG_TC, a, dict(reserve_cand=1)),
                       (wg.WG_TC, b, dict(reserve_full=reserve_mb * MB // 8))])
        _drain(c)
        hs[0].wait()
        assert np.array_equal(hs[0].result(), _closed(*small))
        st = hs[1].wait()
        assert (st.n_tuples, st.iterations, hs[1].digest()) == (n, iters, dg)
        assert hs[1].delta_sizes() == list(log)
        for h in hs:
            h.free()
        # and the context serves on
        h, = c.submit([(wg.WG_TC, a)])
        _drain(c)
        assert np.array_equal(h.result(), _closed(*small))


def test_lane_beside_an_idle_engine():
    # the batch engine of an earlier request holds a third of the budget; a relation
    # loaded after the submission leaves too little for the lane's 112 MB of bit sets
    from paper_2607_17571_gb300 import wg
    first, e, fill = _pairs(5000), _pairs(15_000), _pairs(4_300_000)
    with wg.Context(0, mem_budget=400 * MB, torch_memory=False) as c:
        h, = c.submit([(wg.WG_TC, c.load(*first), dict(reserve_cand=1))])
        h.wait()
        h.free()
        h, = c.submit([(wg.WG_TC, c.load(*e))])
        c.load(*fill)
        assert c.mem_used() > (400 - 112) * MB
        h.wait()
        assert np.array_equal(h.result(), _closed(*e))
