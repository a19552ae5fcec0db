"""Same-generation rows of hubs: a row of more than 256 children is several
items (slices of its children).  Slices that are exactly full, hubs of one and
of several parents, hubs that get new tuples at several iterations (cycles back
to their parents), beside small rows, single and submitted.  Exact equality
with the oracle and with the sorted-array pipeline."""
import numpy as np
import pytest

from oracle import oracle_sg
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _hub(kids, parents, back):
    """Roots 0 (and 3) above a hub 1 and a vertex of few children; with `back` two
    children of the hub lead to a root again."""
    e = [(0, 1), (0, 2), (2, 5), (2, 6), (2, 7)]
    if parents == 2:
        e += [(3, 1), (3, 4), (4, 8), (4, 9)]
    e += [(1, 100 + i) for i in range(kids)]
    if back:
        e += [(100, 0), (100 + kids // 2, 3)]
    return tuple(np.array(e, dtype=np.uint32).T)


def _outcome(q):
    st = q.poll()
    return st.error, st.n_tuples, st.iterations, st.candidates, q.delta_sizes(), q.result()


def _same(got, want):
    for g in got[1:]:
        assert g[:5] == got[0][:5]
    for g in got:
        assert g[:3] == (0, want.keys.shape[0], want.iters) and g[4] == want.log.tolist()
        assert np.array_equal(g[5], want.keys)


@pytest.mark.parametrize("kids", [255, 256, 257, 512, 513, 2049])
@pytest.mark.parametrize("parents,back", [(1, False), (2, False), (1, True), (2, True)])
def test_hub(kids, parents, back):
    from paper_2607_17571_gb300 import wg
    e = _hub(kids, parents, back)
    want = oracle_sg(*e)
    with wg.Context(0) as c:
        rel = c.load(*e)
        got = []
        for kw in ({}, dict(side_run="never")):
            q = c.sg(rel, **kw)
            q.wait()
            got.append(_outcome(q))
            q.free()
        _same(got, want)
        small = I.sg_forest(700, 4, 2.0, 0.02, kids)
        rels = [c.load(small.src, small.dst), rel, c.load(*_hub(kids + 500, 1, False))]
        hs = c.submit([(wg.WG_SG, r) for r in rels])
        while c.serve_step(16):
            pass
        _same([_outcome(hs[1])], want)
        _same([_outcome(hs[0])], oracle_sg(small.src, small.dst))
        assert hs[2].poll().n_tuples == oracle_sg(*_hub(kids + 500, 1, False)).keys.shape[0]


def test_wide_ranks():
    # 32-bit ranks (among many edges that join nothing), a hub of 79 slices, some of
    # its children with one child each
    from paper_2607_17571_gb300 import wg
    kids, n = 20_000, 3000
    k, pad = np.arange(kids), 400_000 + np.arange(25_000)
    src = np.concatenate([np.zeros(1, int), np.full(kids, 1), 10 + k[:n], pad])
    dst = np.concatenate([np.ones(1, int), 10 + k, 200_000 + k[:n], pad + 100_000])
    with wg.Context(0) as c:
        rel = c.load(src.astype(np.uint32), dst.astype(np.uint32))
        q = c.sg(rel)
        q.wait()
        st = q.poll()
        assert (st.n_tuples, st.iterations) == (kids * (kids - 1) + n * (n - 1), 2)
        assert q.delta_sizes() == [kids * (kids - 1), n * (n - 1), 0]
        assert st.candidates == kids * (kids - 1) + n * (n - 1)
        q.free()
