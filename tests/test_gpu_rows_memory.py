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
