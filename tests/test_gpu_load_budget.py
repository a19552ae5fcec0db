"""What the row fixpoints keep beside a relation is optional: a budget that holds
the relations themselves holds them loaded, queries on them are answered, and
the layout comes back once there is room."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MB = 1 << 20


def _pairs(seed, ne):
    """ne disjoint edges: twice as many vertices, where the layout weighs most."""
    ids = np.random.default_rng(seed).choice(1 << 24, size=2 * ne, replace=False).astype(np.uint32)
    return ids[:ne], ids[ne:]


def _closure(src, dst):
    return np.sort((src.astype(np.uint64) << np.uint64(32)) | dst)


@pytest.mark.parametrize("count", [1, 12])
def test_relations_that_fit_without_layouts_load(count):
    from paper_2607_17571_gb300 import wg
    ne = 150_000
    # resident: 8-byte keys and 4-byte successors per edge, offset and id per
    # vertex; while loading: input, sort scratch and copies, under 32 bytes per edge
    budget = count * (12 * ne + 8 * 2 * ne + 8192) + 32 * ne + MB
    with wg.Context(0, mem_budget=budget, torch_memory=False) as c:
        es = [_pairs(k, ne) for k in range(count)]
        rels = [c.load(*e) for e in es]
        for e, r in zip(es, rels):
            assert r.info() == dict(n_edges=ne, n_vertices=2 * ne, field_bits=19)
            assert c.triangles(r) == 0
        assert c.mem_used() <= budget


def test_layout_returns_with_room():
    from paper_2607_17571_gb300 import wg
    first = _pairs(0, 2000)

    def closure(c, rel):
        q = c.tc(rel)
        q.wait()
        assert np.array_equal(q.result(), _closure(*first))
        n = q.poll().gpu_launches
        q.free()
        return n

    with wg.Context(0, mem_budget=48 * MB, torch_memory=False) as c:
        rel = c.load(*first)
        rows = closure(c, rel)
        fill = []
        with pytest.raises(wg.WgError):  # until nothing more fits: no layout is left
            while True:
                fill.append(c.load(*_pairs(len(fill) + 1, 2000)))
        for f in fill[::2]:  # room for a query, not for everything
            f.free()
        closure(c, rel)
        for f in fill[1::2]:
            f.free()
        assert closure(c, rel) == rows
        rel.free()
