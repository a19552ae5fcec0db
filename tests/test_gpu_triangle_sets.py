"""Triangle counting by set intersection at the sizes where it can go wrong: bit
sets that end mid-word, each CTA shape, neighbour lists around a warp's 32, both
ends of an edge taking the count (lists shorter, equal and longer), and the
vertex count past which the join with a binary search takes over.  Exact."""
import numpy as np
import pytest

from oracle import oracle_triangles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c


def _check(ctx, src, dst):
    src, dst = np.asarray(src, np.uint32), np.asarray(dst, np.uint32)
    rel = ctx.load(src, dst)
    assert ctx.triangles(rel) == oracle_triangles(src, dst, n_threads=8)
    rel.free()


@pytest.mark.parametrize("out_deg,in_deg", [(1, 1), (2, 1), (1, 2), (31, 32), (32, 32), (33, 32),
                                            (64, 3), (3, 65), (200, 200)])
def test_list_lengths_around_one_edge(ctx, out_deg, in_deg):
    # edge a -> b; out_deg successors of b, in_deg predecessors of a, sharing
    # the smaller number of vertices (and shifted by one, sharing one less)
    for shift in (0, 1):
        c = np.arange(10, 10 + out_deg)
        d = np.arange(10 + shift, 10 + shift + in_deg)
        _check(ctx, np.concatenate([[0], np.full(out_deg, 1), d]),
               np.concatenate([[1], c, np.full(in_deg, 0)]))


# bit sets of 1 to 47,000 words: 64, 128, 256, 512 and 1,024 threads per CTA; the
# last two counts lie on either side of the limit
@pytest.mark.parametrize("nv", [33, 20_000, 100_000, 250_000, 500_000, 900_000, 1_499_999, 1_500_002])
def test_vertex_counts(ctx, nv):
    rng = np.random.default_rng(nv)
    i = np.arange(nv, dtype=np.int64)
    # a ring (every vertex occurs), triangles across its ends, random edges in a
    # dense core and a loop
    core = rng.choice(nv, size=min(nv, 300), replace=False)
    s, d = core[rng.integers(0, len(core), 6000)], core[rng.integers(0, len(core), 6000)]
    _check(ctx, np.concatenate([i, s, [nv - 1, nv - 2, 0, 5]]),
           np.concatenate([(i + 1) % nv, d, [0, nv - 1, nv - 2, 5]]))
