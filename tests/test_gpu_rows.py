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


@pytest.mark.parametrize("deg", [1, 6, 7, 8, 9, 11, 12, 15, 16, 31, 39, 40, 71, 1023, 1024, 1025, 3000])
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


def _small_rows_graph(nv, seed):
    """nv vertices, most reaching few others; chains, stars and hubs whose rows
    have 254 to 258 tuples (the small rows end at 256), a few rows of thousands
    and one cycle."""
    rng = np.random.default_rng(seed)
    s, d = [np.arange(0, nv - 1, 2)], [np.arange(1, nv, 2)]
    at = nv // 2
    for n in (254, 255, 256, 257, 258):
        chain = np.arange(at, at + n + 1)           # rows of n, n - 1, ... tuples
        s.append(chain[:-1]); d.append(chain[1:])
        at += n + 1
        s.append(np.full(n, at)); d.append(np.arange(at + 1, at + 1 + n))  # a star of n leaves
        at += n + 1
    s.append(np.full(3000, at)); d.append(rng.integers(0, nv, 3000))
    s.append(np.arange(20, 140)); d.append(np.arange(21, 141) % 140 + (np.arange(21, 141) >= 140) * 20)
    s.append(rng.integers(0, nv, nv // 3)); d.append(rng.integers(0, nv, nv // 3))
    return np.concatenate(s), np.concatenate(d)


# bit sets of 8 to 96 KB (each CTA shape), the widest relation that has them and
# the narrowest that has none
@pytest.mark.parametrize("nv", [65_538, 140_000, 262_146, 300_000, 786_432, 786_434])
def test_small_rows_apart(ctx, nv):
    _check(ctx, *_small_rows_graph(nv, nv))


@pytest.mark.parametrize("cap", [1, 3, 64, 255, 256, 257])
def test_small_rows_iteration_caps(ctx, cap):
    _check(ctx, *_small_rows_graph(70_000, 5), max_iters=cap)


@pytest.mark.parametrize("rows,budget_mb", [(9000, 6000), (9000, 1900), (26_000, 1900)])
def test_long_rows_and_the_budget(rows, budget_mb):
    # rows of 261 tuples over 400,000 vertices need bit sets of 50 KB each.  A
    # quarter of the budget holds them; or it does not and they are made room
    # for when they turn up; or they do not fit at all (1.3 GB beside the small
    # rows' 0.4) and the sorted-array pipeline takes the query
    from oracle import oracle_tc_reach
    from paper_2607_17571_gb300 import wg
    i, hubs = np.arange(rows), np.arange(30_000, 30_010)
    src = np.concatenate([np.arange(0, 400_000, 2), i, np.repeat(hubs, 260)]).astype(np.uint32)
    dst = np.concatenate([np.arange(1, 400_001, 2), 30_000 + i % 10,
                          np.tile(np.arange(50_000, 50_260), 10)]).astype(np.uint32)
    n, iters, log, dg = oracle_tc_reach(src, dst, n_threads=8)
    with wg.Context(0, mem_budget=budget_mb << 20) as c:
        rel = c.load(src, dst)
        for _ in range(2):
            q = c.tc(rel)
            st = q.wait()
            assert (st.n_tuples, st.iterations, q.digest()) == (n, iters, dg)
            assert q.delta_sizes() == list(log)
            q.free()


@pytest.mark.parametrize("n", [63, 64, 65, 66, 95, 96, 97, 129, 161])
@pytest.mark.parametrize("wide", [0, 5_000, 70_000])
def test_iterations_past_the_shared_log(ctx, n, wide):
    """A path of n edges, alone (one warp a row) and beside wide single edges (more
    warps, 32-bit ranks): its iterations past 64 are logged 32 at a time."""
    g = I.path(n + 1)
    at = int(max(g.src.max(), g.dst.max())) + 1
    b = np.arange(at, at + wide, dtype=np.uint32)
    _check(ctx, np.concatenate([g.src, b[0::2]]), np.concatenate([g.dst, b[1::2]]))
