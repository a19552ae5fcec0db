"""The merge-path forms of wg_unique_diff and wg_merge_disjoint at the edges of
their tiles and of the rule that picks them: tiles that end mid-way, one side
exhausted, runs of duplicates across tiles, duplicates in the full relation, the
largest key, and full relations around 64 times the candidates (past which each
key is searched).  Exact, against numpy."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DT = {4: np.uint32, 8: np.uint64}


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c


def _dev(a):
    t = torch.from_numpy(a.view(np.int32 if a.itemsize == 4 else np.int64)).cuda()
    torch.cuda.synchronize()
    return t


def _diff(ctx, cand, full, kb):
    tc, tf = _dev(cand), _dev(full)
    out = torch.empty_like(tc)
    m = ctx.unique_diff(tc.data_ptr(), len(cand), tf.data_ptr(), len(full), out.data_ptr(), kb)
    want = np.setdiff1d(cand, full)
    assert m == len(want) and np.array_equal(out.cpu().numpy().view(DT[kb])[:m], want)


@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("n,nf", [(1, 1), (1, 64), (1, 65), (2, 4095), (1000, 1048), (2047, 1), (2048, 2048),
                                  (4097, 4095), (5000, 320_000), (5000, 320_001), (300_000, 10_000)])
def test_unique_diff(ctx, kb, n, nf):
    rng = np.random.default_rng(n * 3 + nf)
    top = np.iinfo(DT[kb]).max
    for hi in (max(2, (n + nf) // 3), 4 * (n + nf), int(top)):
        cand = np.sort(rng.integers(0, hi, n, dtype=DT[kb], endpoint=True))
        full = np.sort(rng.integers(0, hi, nf, dtype=DT[kb], endpoint=True))  # (with duplicates)
        full[: nf // 3] = rng.choice(cand, nf // 3)
        full.sort()
        _diff(ctx, cand, full, kb)
    same = np.full(n, top, DT[kb])                 # one run over every tile, the largest key
    _diff(ctx, same, np.sort(rng.integers(0, 1000, nf, dtype=DT[kb])), kb)
    _diff(ctx, same, np.append(np.zeros(nf - 1, DT[kb]), same[:1]), kb)
    lo = np.arange(n, dtype=DT[kb])                # all candidates before or after full
    hi = lo[-1] + 1 + np.arange(nf, dtype=DT[kb])
    _diff(ctx, lo, hi, kb)
    _diff(ctx, lo + DT[kb](nf), np.arange(nf, dtype=DT[kb]), kb)


@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("na,nb", [(1, 4095), (15, 1), (16, 17), (2048, 2048), (4095, 4097), (4096, 4096),
                                   (100_000, 3), (70_000, 130_001)])
def test_merge(ctx, kb, na, nb):
    rng = np.random.default_rng(na + nb)
    u = np.unique(rng.integers(0, np.iinfo(DT[kb]).max, 2 * (na + nb) + 9, dtype=DT[kb], endpoint=True))
    pick = rng.permutation(len(u))[: na + nb]
    whole = np.sort(u[pick])
    whole[-1] = np.iinfo(DT[kb]).max
    inter = np.zeros(na + nb, bool)
    inter[rng.permutation(na + nb)[:na]] = True
    for mask in (inter, np.arange(na + nb) < na, np.arange(na + nb) >= nb):  # mixed, a first, b first
        a, b = _dev(whole[mask]), _dev(whole[~mask])
        out = torch.empty(na + nb, dtype=a.dtype, device="cuda")
        ctx.merge_disjoint(a.data_ptr(), na, b.data_ptr(), nb, out.data_ptr(), kb)
        assert np.array_equal(out.cpu().numpy().view(DT[kb]), whole)
