"""TC over relations wide enough (more than 2^18 vertices, many rows of more than 256
tuples) that a sample of the long rows decides between rows and the sorted-array
pipeline: deep ones go to the pipeline, shallow ones stay, both give the closure."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _paths(p, n, hub=0):
    """p disjoint paths of n vertices; `hub`: every vertex also points to one vertex
    with that many leaves."""
    i = np.arange(p * n)
    s, d = i[i % n != n - 1], i[i % n != n - 1] + 1
    if hub:
        h = p * n
        s = np.concatenate([s, i, np.full(hub, h)])
        d = np.concatenate([d, np.full(p * n, h), h + 1 + np.arange(hub)])
    return s.astype(np.uint32), d.astype(np.uint32)


def _fans(rows, hubs, leaves):
    """`rows` sources, each pointing to one of `hubs` vertices with `leaves` leaves."""
    i, h = np.arange(rows), rows + np.arange(hubs)
    leaf = rows + hubs + np.arange(hubs * leaves)
    return (np.concatenate([i, np.repeat(h, leaves)]).astype(np.uint32),
            np.concatenate([rows + i % hubs, leaf]).astype(np.uint32))


def _run(c, rel, **kw):
    q = c.tc(rel, **kw)
    st = q.wait()
    got = (st.n_tuples, st.iterations, st.candidates, q.delta_sizes(), q.digest())
    n = st.gpu_launches
    q.free()
    return got, n


@pytest.mark.parametrize("case", ["paths", "paths_to_a_hub", "fans", "mixed", "capped"])
def test_sampled(case):
    from paper_2607_17571_gb300 import wg
    e = {"paths": lambda: _paths(1300, 400),          # 187,000 rows of 257 to 399 tuples
         "capped": lambda: _paths(1300, 400),
         "paths_to_a_hub": lambda: _paths(700, 400, 300),  # every row starts wide, then deep
         "fans": lambda: _fans(60_000, 900, 300),     # 60,000 rows of 301 tuples, two levels
         "mixed": lambda: _fans(50_000, 900, 290)}[case]()
    if case == "mixed":  # some deep rows among many shallow ones
        p = _paths(30, 900)
        e = tuple(np.concatenate([a, b + np.uint32(400_000)]) for a, b in zip(e, p))
    kw = dict(max_iters=300) if case == "capped" else {}
    with wg.Context(0) as c:
        rel = c.load(*e)
        if case == "capped":
            for more in ({}, dict(reserve_cand=1)):
                q = c.tc(rel, **kw, **more)
                with pytest.raises(wg.WgError):
                    q.wait()
                st = q.poll()
                assert (st.n_tuples, st.iterations) == (1300 * sum(399 - k for k in range(301)), 300)
                assert q.delta_sizes() == [1300 * (399 - k) for k in range(301)]
                q.free()
            return
        want, _ = _run(c, rel, reserve_cand=1)  # the pipeline
        for _ in range(2):
            got, launches = _run(c, rel)
            assert got == want
            # (the pipeline: some ten kernels an iteration)
            assert (launches > 1000) == case.startswith("paths")
        if case == "paths":
            assert want[:3] == (1300 * 400 * 399 // 2, 399, 1300 * 400 * 399 // 2)


def test_deep_without_room_for_the_pipeline():
    # the reserve of 14 GB is one buffer of the rows' (11 GB of lists and bit sets beside
    # it) and two of the pipeline's: a deep query that does not fit there is run by
    # rows after all
    from paper_2607_17571_gb300 import wg
    p, n = 800, 500
    with wg.Context(0, torch_memory=False) as c:
        want, launches = _run(c, c.load(*_paths(p, n)))
        assert launches > 1000
    with wg.Context(0, mem_budget=26_000 << 20, torch_memory=False) as c:
        got, launches = _run(c, c.load(*_paths(p, n)), reserve_full=(14 << 30) // 8)
        assert got == want and launches < 1000


@pytest.mark.parametrize("budget_mb", [4500, 6000, 11_000, 14_000])
def test_deep_under_budgets(budget_mb):
    # what the pipeline grows through, the lists and a sample, or all of the bit sets
    from paper_2607_17571_gb300 import wg
    p, n = 800, 500
    with wg.Context(0, mem_budget=budget_mb << 20, torch_memory=False) as c:
        got, _ = _run(c, c.load(*_paths(p, n)))
        assert got[:4] == (p * n * (n - 1) // 2, n - 1, p * n * (n - 1) // 2,
                           [p * (n - 1 - k) for k in range(n)])
        h, = c.submit([(wg.WG_TC, c.load(*_paths(p, n)))])  # as a served large request
        while c.serve_step(16):
            pass
        assert (h.wait().n_tuples, h.delta_sizes()) == (got[0], got[3])
