"""Same-generation over rows of bit sets (the path a plain wg_sg takes) against
the oracle and the sorted-array pipeline, where it can go wrong: rows that end
mid-piece, vertices of one and of several parents, self-loops and cycles, hubs,
rows of one and of 32 mask words, both rank widths and the widest relation,
iteration caps, instances that end at different iterations in one launch, and a
result buffer that grows.  Exact equality."""
import numpy as np
import pytest

from oracle import oracle_sg
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c


def _outcome(q):
    st = q.poll()
    done = st.error == 0
    return (st.error, st.n_tuples, st.iterations, st.candidates, q.delta_sizes(),
            q.digest() if done else None)


def _check(ctx, src, dst, **opts):
    src, dst = np.asarray(src, np.uint32), np.asarray(dst, np.uint32)
    want = oracle_sg(src, dst, **opts)
    rel = ctx.load(src, dst)
    got = []
    for kw in ({}, dict(side_run="never")):  # rows, the sorted-array pipeline
        q = ctx.sg(rel, **opts, **kw)
        ctx.lib.wg_wait(ctx.h, q.id, 0)
        got.append(_outcome(q))
        if got[-1][0] == 0:
            assert np.array_equal(q.result(), want.keys)
        q.free()
    rel.free()
    assert got[0] == got[1]
    assert got[0][1:3] == (want.keys.shape[0], want.iters) and got[0][4] == want.log.tolist()


@pytest.mark.parametrize("n", [40, 127, 128, 129, 1000, 4095, 4097])
@pytest.mark.parametrize("cross", [0.0, 0.01, 0.2])
def test_forests(ctx, n, cross):
    g = I.sg_forest(n, 5, 2.0, cross, n + int(100 * cross))
    _check(ctx, g.src, g.dst)


@pytest.mark.parametrize("n,m", [(5, 12), (60, 90), (130, 260), (400, 700), (1200, 1500)])
def test_several_parents_loops_and_cycles(ctx, n, m):
    g = I.random_small(n, m, n)
    _check(ctx, g.src, g.dst)
    c = I.cycle(n // 2 + 1)  # two cycles with a common parent
    _check(ctx, np.concatenate([c.src, c.src + 10_000, [90_000, 90_000]]),
           np.concatenate([c.dst, c.dst + 10_000, [0, 10_000]]))


@pytest.mark.parametrize("kids", [7, 8, 9, 33, 700])
def test_hubs(ctx, kids):
    # a root with `kids` children, each with 0 to 9 children
    k = np.arange(1, kids + 1)
    grand = np.repeat(k, k % 10)
    _check(ctx, np.concatenate([np.zeros(kids, int), grand]),
           np.concatenate([k, 10_000 + np.arange(len(grand))]))


@pytest.mark.parametrize("nv", [65_536, 65_537, 131_072, 131_073])
def test_vertex_counts(ctx, nv):
    # many small trees, ids permuted; a few vertices with two parents
    rng = np.random.default_rng(nv)
    i = np.arange(nv)
    child = i[i % 16 != 0]
    src = child // 16 * 16 + (child % 16 - 1) // 2
    ids = rng.permutation(nv)
    extra = rng.integers(0, nv, (40, 2))
    _check(ctx, np.concatenate([ids[src], extra[:, 0]]), np.concatenate([ids[child], extra[:, 1]]))


@pytest.mark.parametrize("cap", [1, 2, 5, 8])
def test_iteration_caps(ctx, cap):
    for g in (I.sg_forest(900, 3, 2.0, 0.02, 4), I.binary_tree(7), I.random_small(100, 160, 3)):
        _check(ctx, g.src, g.dst, max_iters=cap)


def test_batched_instances_end_at_different_iterations():
    from paper_2607_17571_gb300 import wg
    gs = [I.binary_tree(d) for d in (1, 3, 8)] + [I.sg_forest(n, 4, 2.0, 0.01, n) for n in (60, 700, 2500)]
    gs += [I.random_small(80, 140, 9), I.path(30)]
    with wg.Context(0) as c:
        rels = [c.load(g.src, g.dst) for g in gs]
        kinds = [wg.WG_SG] * len(gs) + [wg.WG_TC] * 2
        both = []
        for kw in ({}, dict(side_run="never")):
            hs = c.submit([(k, r, kw) for k, r in zip(kinds, rels + rels[:2])] +
                          [(wg.WG_SG, rels[5], dict(max_iters=3, **kw))])
            while c.serve_step(16):
                pass
            both.append([_outcome(h) for h in hs])
            for h in hs:
                h.free()
        assert both[0] == both[1]
        for g, got in zip(gs, both[0]):
            want = oracle_sg(g.src, g.dst)
            assert got[1:3] == (want.keys.shape[0], want.iters) and got[4] == want.log.tolist()
