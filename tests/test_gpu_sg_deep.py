"""Same-generation fixpoints that take more iterations than the relation has
vertices: two cycles of coprime lengths under one parent meet in lcm(p, q)
levels.  Every per-iteration size against the oracle's log, for queries
run singly, submitted alone or beside others, and past what a query keeps."""
import numpy as np
import pytest

from oracle import oracle_sg
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu
BATCH_LOG = 1024  # per-iteration sizes kept per submitted query


def _cycles(p, q):
    """Two cycles of p and q vertices, one vertex of each a child of a root."""
    a, b = I.cycle(p), I.cycle(q)
    return (np.concatenate([a.src, b.src + 10_000, [90_000, 90_000]]).astype(np.uint32),
            np.concatenate([a.dst, b.dst + 10_000, [0, 10_000]]).astype(np.uint32))


def _same(got, want, keep):
    st = got.poll()
    assert (st.error, st.n_tuples, st.iterations) == (0, want.keys.shape[0], want.iters)
    assert got.delta_sizes() == want.log.tolist()[:keep]
    assert np.array_equal(got.result(), want.keys)


@pytest.mark.parametrize("lengths", [[(3, 4)], [(31, 32)], [(33, 34)],
                                     [(20, 21), (3, 4), (31, 32), (5, 9)], [(33, 34), (2, 3)]])
def test_submitted(lengths):
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        es = [_cycles(p, q) for p, q in lengths]
        tree = I.binary_tree(5)
        es.append((tree.src, tree.dst))
        if len(lengths) == 1:
            es.pop()  # alone
        for kw in ({}, dict(side_run="never")):  # rows, the sorted-array pipeline
            rels = [c.load(*e) for e in es]
            hs = c.submit([(wg.WG_SG, r, kw) for r in rels])
            while c.serve_step(16):
                pass
            for e, h in zip(es, hs):
                _same(h, oracle_sg(*e), BATCH_LOG)
                h.free()
            for r in rels:
                r.free()


@pytest.mark.parametrize("p,q", [(2, 3), (3, 4), (20, 21), (31, 32), (40, 41), (256, 257)])
def test_single(p, q):
    from paper_2607_17571_gb300 import wg
    e = _cycles(p, q)
    want = oracle_sg(*e)  # (256 * 257 = 65,792 iterations: more than a query keeps)
    with wg.Context(0) as c:
        for kw in ({}, dict(side_run="never")):
            rel = c.load(*e)
            h = c.sg(rel, **kw)
            h.wait()
            _same(h, want, 1 << 16)
            h.free()
            rel.free()


def test_iterations_past_2_to_32_arrivals():
    # every row listed at the start: a full grid of CTAs meets at each of 1,770,230
    # barriers.  Coprime cycles: each vertex of one with each of the other, two new
    # tuples an iteration
    from paper_2607_17571_gb300 import wg
    p, q = 1330, 1331
    with wg.Context(0) as c:
        rel = c.load(*_cycles(p, q))
        h = c.sg(rel, max_iters=1 << 22)
        h.wait()
        st = h.poll()
        assert (st.n_tuples, st.iterations) == (2 * p * q, p * q)
        assert h.delta_sizes() == [2] * (1 << 16)
        a, b = np.arange(p, dtype=np.uint64), np.arange(q, dtype=np.uint64) + np.uint64(10_000)
        ab = (a[:, None] << np.uint64(32) | b).ravel()
        ba = (b[:, None] << np.uint64(32) | a).ravel()
        assert np.array_equal(h.result(), np.concatenate([ab, ba]))
        h.free()
