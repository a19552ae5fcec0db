"""Device memory of a plain TC query over a wide, sparse relation: lists for the
rows and bit sets for the rows that need one, not for every row."""
import numpy as np
import pytest

from oracle import oracle_tc
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,edges", [(100_000, 60_000), (100_000, 90_000)])
def test_bit_sets_of_the_long_rows_only(nodes, edges):
    from paper_2607_17571_gb300 import wg
    g = I.er_graph(nodes, edges, 7)
    want = oracle_tc(g.src, g.dst)
    rows = np.bincount((want.keys >> np.uint64(32)).astype(np.int64))
    with wg.Context(0, mem_budget=8 << 30, torch_memory=False) as c:
        rel = c.load(g.src, g.dst)
        nv, before = rel.info()["n_vertices"], c.mem_used()
        for _ in range(2):  # a new engine, and one that has bit sets already
            q = c.tc(rel)
            q.wait()
            assert q.delta_sizes() == want.log.tolist()
            assert np.array_equal(q.result(), want.keys)
            long_rows = int((rows > 256).sum())
            # 1 KB of list and 12 bytes of bookkeeping a vertex, a bit set a long
            # row (and an eighth more), the result's reserve, 8 MB besides
            most = (nv * (1024 + 12) + (long_rows * 9 // 8 + 64) * (nv // 8 + 16) +
                    max(4 * edges, 2 * want.keys.shape[0]) * 8 + (8 << 20))
            assert c.mem_used() - before <= most
            q.free()


def _long_rows(rows):
    """`rows` rows of 261 tuples over 400,000 vertices."""
    i, hubs = np.arange(rows), np.arange(30_000, 30_010)
    src = np.concatenate([np.arange(0, 400_000, 2), i, np.repeat(hubs, 260)]).astype(np.uint32)
    dst = np.concatenate([np.arange(1, 400_001, 2), 30_000 + i % 10,
                          np.tile(np.arange(50_000, 50_260), 10)]).astype(np.uint32)
    return src, dst


def test_a_passing_shortage_marks_no_relation():
    # 26,000 bit sets take 1.4 GB beside 0.4 GB of lists: too much while another
    # query's result (0.5 GB) is held, and room enough once it is freed
    from oracle import oracle_tc_reach
    from paper_2607_17571_gb300 import wg
    src, dst = _long_rows(26_000)
    n, iters, log, dg = oracle_tc_reach(src, dst, n_threads=8)
    g = I.er_graph(12_000, 36_000, 3)
    with wg.Context(0, mem_budget=2250 << 20, torch_memory=False) as c:
        rel, other = c.load(src, dst), c.load(g.src, g.dst)

        def launches():
            q = c.tc(rel)
            st = q.wait()
            assert (st.n_tuples, st.iterations, q.digest()) == (n, iters, dg)
            k = st.gpu_launches
            q.free()
            return k

        held = c.tc(other)
        held.wait()
        assert launches() > 20   # the sorted-array pipeline: some ten kernels an iteration
        held.free()
        other.free()
        assert launches() < 20   # rows again


@pytest.mark.parametrize("budget_mb", range(1730, 1830, 10))
def test_result_that_does_not_fit_beside_the_bit_sets(budget_mb):
    # lists and bit sets take some 1,743 MB, the result 50 MB more
    from oracle import oracle_tc_reach
    from paper_2607_17571_gb300 import wg
    src, dst = _long_rows(26_000)
    n, iters, log, dg = oracle_tc_reach(src, dst, n_threads=8)
    with wg.Context(0, mem_budget=budget_mb << 20, torch_memory=False) as c:
        q = c.tc(c.load(src, dst))
        st = q.wait()
        assert (st.n_tuples, st.iterations, q.digest()) == (n, iters, dg)
        assert q.delta_sizes() == list(log)
