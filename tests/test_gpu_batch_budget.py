"""The budget cases of submitted queries (preemption, growths that fail at every
step, hopeless and exclusive requests) on the batch engines: plain small queries
run on row lanes, so the same cases are run with every request, or every other
one, asking for candidate buffers, which takes it to the batch engine of its key
class."""
import numpy as np
import pytest

import test_gpu_batch as batch
from oracle import oracle_tc
from paper_2607_17571_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[1, 2], ids=["engines", "engines_and_lanes"])
def engines(request, monkeypatch):
    from paper_2607_17571_gb300 import wg
    submit = wg.Context.submit

    def routed(self, reqs):
        out = []
        for i, r in enumerate(reqs):
            opts = dict(r[2]) if len(r) > 2 else {}
            if i % request.param == 0:
                opts["reserve_cand"] = 1
            out.append((r[0], r[1], opts))
        return submit(self, out)

    monkeypatch.setattr(wg.Context, "submit", routed)
    return request.param


def test_preemption(engines):
    batch.test_preemption_under_small_budget()


def test_larger_than_budget(engines):
    batch.test_query_larger_than_budget_fails_cleanly()


def test_hopeless_large_request(engines):
    batch.test_hopeless_large_request_fails_beside_small_ones()


@pytest.mark.parametrize("budget_mb", [72, 96, 128, 160, 200, 256, 320])
def test_failed_growth(engines, budget_mb):
    batch.test_failed_growth_leaves_engines_whole(budget_mb)


@pytest.mark.parametrize("big_kind", ["batch", "solo"])
@pytest.mark.parametrize("budget_mb", [96, 128, 192])
def test_fits_alone(engines, budget_mb, big_kind):
    if engines == 1:
        batch.test_query_that_fits_alone_completes_in_a_mix(budget_mb, big_kind)
        return
    # lanes end their requests early, and their results, not yet taken, may leave too
    # little for the large one (or for an engine's first pools): every request ends
    from paper_2607_17571_gb300 import wg
    big, smalls, want_big, want_smalls = batch._exclusive_cases(big_kind)
    with wg.Context(0, mem_budget=budget_mb << 20) as c:
        rels = [c.load(g.src, g.dst) for g in smalls[:4] + [big] + smalls[4:]]
        want = want_smalls[:4] + [want_big] + want_smalls[4:]
        done = 0
        for h, w in zip(c.submit([(wg.WG_TC, r) for r in rels]), want):
            try:
                h.wait()
                assert np.array_equal(h.result(), w.keys)
                done += 1
            except wg.WgError as e:
                assert e.code in (wg.WG_E_BUDGET, wg.WG_E_NOMEM)
            h.free()
        assert done >= 4  # those on lanes at least
        last = I.er_graph(300, 700, 17)  # everything is free again: an engine holds it
        h, = c.submit([(wg.WG_TC, c.load(last.src, last.dst))])
        h.wait()
        assert np.array_equal(h.result(), oracle_tc(last.src, last.dst).keys)
        h.free()


def test_mix_and_caps(engines, ctx):
    batch.test_alone_equals_mix_equals_oracle(ctx)
    batch.test_slot_reuse_with_running_neighbours(ctx)
    batch.test_iteration_cap_in_batch(ctx)


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c
