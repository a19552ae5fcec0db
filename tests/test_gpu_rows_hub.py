"""TC over relations with one heavy source: a row is one CTA's work, so a hub whose
two-paths outweigh everything else runs on the sorted-array pipeline, and the
same hub among enough other work, or a light one, by rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _hub(m, n, pairs=0):
    """A source of m children with the same n children each, and disjoint edges."""
    mid, leaf, p = 1 + np.arange(m), 1 + m + np.arange(n), 10**6 + np.arange(pairs)
    return (np.concatenate([np.zeros(m, int), np.repeat(mid, n), p]).astype(np.uint32),
            np.concatenate([mid, np.tile(leaf, m), p + 10**6]).astype(np.uint32))


def _run(c, rel, **kw):
    q = c.tc(rel, **kw)
    st = q.wait()
    got = (st.n_tuples, st.iterations, st.candidates, q.delta_sizes(), q.digest())
    k = st.gpu_launches
    q.free()
    return got, k


# (launches: rows take 4 to 12 kernels, the pipeline some ten an iteration)
@pytest.mark.parametrize("m,n,pairs,rows", [
    (2000, 2000, 0, False), (500, 15_000, 0, False), (100, 60_000, 0, False),
    (1000, 5000, 40_000, False),   # 32-bit ranks
    (650, 650, 0, True), (680, 680, 0, False),  # about 440,000 edges: the line
    (3000, 3000, 100_000, True),   # 17-bit ranks, where the pipeline starts slowly
    (300, 3000, 100_000, True)])
def test_routes(m, n, pairs, rows):
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        rel = c.load(*_hub(m, n, pairs))
        want, k = _run(c, rel, reserve_cand=1)  # the pipeline
        assert want[:2] == (m + n + m * n + pairs, 2) and want[2] == 2 * m * n + m + pairs
        for _ in range(2):
            got, launches = _run(c, rel)
            assert got == want and (launches < 15) == rows
        q = c.tc(rel, max_iters=1)
        st = q.poll()
        while st.state == wg.WG_RUNNING:
            st = q.poll()
        assert st.iterations == want[1] - 1 and q.delta_sizes() == want[3][:2]
        q.free()


@pytest.mark.parametrize("reserve", [0, (500 << 20) // 4])
def test_hub_without_room_for_the_pipeline(reserve):
    # the pipeline starts with more than 900 MB for 4 million edges (and two buffers of
    # the reserve): by rows after all
    from paper_2607_17571_gb300 import wg
    e = _hub(2000, 2000)
    with wg.Context(0) as c:
        want, _ = _run(c, c.load(*e), reserve_cand=1)
    with wg.Context(0, mem_budget=900 << 20, torch_memory=False) as c:
        rel = c.load(*e)
        got, launches = _run(c, rel, reserve_full=reserve)
        assert got == want and launches < 15
        h, = c.submit([(wg.WG_TC, rel, dict(reserve_full=reserve))])
        while c.serve_step(16):
            pass
        assert (h.wait().n_tuples, h.delta_sizes(), h.digest()) == (want[0], want[3], want[4])
