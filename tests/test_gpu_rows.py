"""Transitive closure row by row (the path a plain wg_tc takes) against the
oracle and against the sorted-array pipeline, at the sizes where the rows can
go wrong: bit-set words and 16-byte vectors that end mid-way, 16- and 32-bit
ranks, adjacency records that are exactly full or overflow, rows longer than
the list kept in shared memory, more levels than are counted there, iteration
caps, and a result buffer that is too small at first.  Exact equality."""
import numpy as np
import pytest

from oracle import oracle_tc
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _pairs(nv, extra):
    """nv vertices in disjoint edges i -> i + nv/2, plus the edges `extra`."""
    h = nv // 2
    a = np.arange(nv - h, dtype=np.int64)
    src, dst = a, np.minimum(a + h, nv - 1)
    e = np.array(extra, dtype=np.int64).reshape(-1, 2)
    return np.concatenate([src, e[:, 0]]), np.concatenate([dst, e[:, 1]])


def _star(deg, tail):
    """0 -> 1..deg, and each of the first `tail` leaves into a chain of 3."""
    e = [(0, i) for i in range(1, deg + 1)]
    for i in range(1, tail + 1):
        e += [(i, deg + 2 * i), (deg + 2 * i, deg + 2 * i + 1)]
    return np.array(e, dtype=np.int64).T


def _check(ctx, src, dst, **opts):
    src, dst = np.asarray(src, np.uint32), np.asarray(dst, np.uint32)
    cap = {k: v for k, v in opts.items() if k == "max_iters"}
    want = oracle_tc(src, dst, **cap)
    rel = ctx.load(src, dst)
    got = []
    for kw in ({}, dict(side_run="never")):  # row by row, the sorted-array pipeline
        q = ctx.tc(rel, **opts, **kw)
        rc = ctx.lib.wg_wait(ctx.h, q.id, 0)
        st = q.poll()
        assert rc == st.error
        keys = q.result() if rc == 0 else None
        got.append((rc, st.n_tuples, st.iterations, st.candidates, q.delta_sizes()))
        if keys is not None:
            assert np.array_equal(keys, want.keys)
        q.free()
    rel.free()
    assert got[0] == got[1]
    assert got[0][1:3] == (want.keys.shape[0], want.iters) and got[0][4] == want.log.tolist()


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c


@pytest.mark.parametrize("nv", [2, 31, 32, 33, 127, 128, 129, 255, 256, 257, 4095, 65535, 65536,
                                65537, 70001])
def test_vertex_counts(ctx, nv):
    top = nv - 1
    _check(ctx, *_pairs(nv, [(top, 0), (0, 1 % nv), (top, top)]))


@pytest.mark.parametrize("deg", [1, 6, 7, 8, 9, 31, 38, 39, 40, 71, 1023, 1024, 1025, 3000])
def test_degrees(ctx, deg):
    _check(ctx, *_star(deg, min(deg, 40)))
    # the hub reached from others, itself among its own successors
    s, d = _star(deg, min(deg, 5))
    _check(ctx, np.append(s, [1, 2 % (deg + 1)]), np.append(d, [0, 0]))


def test_degree_of_every_vertex(ctx):
    # out-degree 65,536 (more than a 16-bit field holds) with 16-bit ranks
    d = np.arange(65536)
    _check(ctx, np.append(np.zeros(65536, int), 5), np.append(d, 0))


@pytest.mark.parametrize("n", [1023, 1025, 3000])
def test_long_rows(ctx, n):
    # strongly connected: every row reaches n vertices; and a cycle with more
    # levels than are counted in shared memory
    g = I.er_graph(n, 4 * n, n)
    _check(ctx, g.src, g.dst)
    g = I.cycle(n // 10)
    _check(ctx, g.src, g.dst)


@pytest.mark.parametrize("cap", [1, 2, 63, 64, 65, 150])
def test_iteration_caps(ctx, cap):
    for g in (I.path(151), I.cycle(66), I.er_graph(300, 900, 3)):
        _check(ctx, g.src, g.dst, max_iters=cap)


def test_result_buffer_grows_and_the_engine_is_reused():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        for g in (I.er_graph(900, 2700, 31), I.path(40), I.er_graph(1000, 3500, 32)):
            want = oracle_tc(g.src, g.dst)
            rel = c.load(g.src, g.dst)
            for _ in range(2):
                q = c.tc(rel, reserve_full=1)
                q.wait()
                assert np.array_equal(q.result(), want.keys)
                assert q.delta_sizes() == want.log.tolist()
                q.free()
            rel.free()


def _drain(ctx):
    while ctx.serve_step(16):
        pass


def test_batched_rows_equal_the_batched_pipeline():
    """Submitted queries row by row (rows of many relations of both rank widths
    in one launch, chunks of 256 rows that end mid-way, iteration caps, more
    iterations than the batch keeps sizes of) against the same queries on the
    batch engines' sorted-array pipeline, and a query freed while it runs."""
    from paper_2607_17571_gb300 import wg
    gs = [I.path(1100), I.path(2), I.er_graph(255, 500, 1), I.er_graph(700, 1500, 2),
          I.er_graph(70_000, 60_000, 3), I.cycle(257), I.rmat_dag(11, 5000, 4),
          I.er_graph(80_000, 50_000, 5), I.path(300)]
    caps = [0, 0, 0, 3, 0, 100, 0, 2, 64]
    with wg.Context(0) as c:
        rels = [c.load(g.src, g.dst) for g in gs]
        got = []
        for kw in ({}, dict(side_run="never")):
            hs = c.submit([(wg.WG_TC, r, dict(max_iters=m, **kw)) for r, m in zip(rels, caps)])
            extra = c.submit([(wg.WG_TC, rels[3], kw)])[0]
            c.serve_step(1)
            extra.free()
            _drain(c)
            assert sorted(c.take_completed()) == sorted(h.id for h in hs)
            out = []
            for h in hs:
                st = h.poll()
                out.append((st.state, st.error, st.n_tuples, st.iterations, st.candidates,
                            h.delta_sizes(), h.digest() if st.state == wg.WG_DONE else None))
                h.free()
            got.append(out)
        assert got[0] == got[1]
        for r in rels:
            r.free()
