"""wg_sort_keys of arrays large enough for the top-digit-first form, where it can go
wrong: the first size that takes it, ragged tails, one to many bits below the top
digit, bins around the most one holds, and keys that must fall back to the
lookback passes (skewed by the sample, or only by the exact count), with an odd
and an even number of passes; and another primitive after each.  Exact, against
torch.sort of the same bit patterns in unsigned order."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
MIN = 1 << 23
SIGN = -(1 << 63)


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_17571_gb300 import wg
    with wg.Context(0) as c:
        yield c


def _sort(ctx, a, bits):
    kb = a.element_size()
    t = a.clone()
    want = (a ^ SIGN).sort().values ^ SIGN if kb == 8 else (a.long() & 0xFFFFFFFF).sort().values.int()
    torch.cuda.synchronize()
    ctx.sort_keys(t.data_ptr(), a.numel(), kb, bits)
    assert torch.equal(t, want)
    # the control block is clear: the next primitive does its work
    out = torch.empty_like(t)
    m = ctx.unique_diff(t.data_ptr(), a.numel(), 0, 0, out.data_ptr(), kb)
    assert torch.equal(out[:m], torch.unique_consecutive(want))


def _uniform(n, kb, bits, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randint(0, 1 << min(bits, 62), (n,), generator=g, device="cuda")
    if bits > 62:
        v = (v << (bits - 62)) | (v & ((1 << (bits - 62)) - 1))
    return v if kb == 8 else v.int()


@pytest.mark.parametrize("kb,bits", [(4, 32), (8, 12), (8, 19), (8, 20), (8, 34), (8, 35), (8, 64)])
@pytest.mark.parametrize("n", [MIN - 1, MIN, MIN + 16_385])
def test_uniform(ctx, kb, bits, n):
    _sort(ctx, _uniform(n, kb, bits, n + bits), bits)


@pytest.mark.parametrize("n", [10_300_001, 20_600_000, 41_000_003, 82_000_000])
def test_more_bins(ctx, n):
    _sort(ctx, _uniform(n, 8, 40, n), 40)


@pytest.mark.parametrize("bits", [33, 48])
def test_skewed_keys_fall_back(ctx, bits):
    n = MIN + 777
    a = _uniform(n, 8, bits, 1)
    _sort(ctx, a & ((1 << (bits - 6)) - 1), bits)   # top bits all zero: the sample sees it
    _sort(ctx, a[:1].repeat(n), bits)               # one key
    up = a.sort().values
    _sort(ctx, up, bits)                            # sorted, reversed (even bins)
    _sort(ctx, up.flip(0), bits)
    # 11 top bits, 4,096 keys a bin; bin 5 gets `held` keys -- few enough for the
    # sample -- around the 8,192 that fit
    sh = bits - 11
    rest = (1 << sh) - 1
    was = ((a >> sh) == 5).nonzero().flatten()
    other = ((a >> sh) != 5).nonzero().flatten()
    for held in (8_000, 8_191, 8_192, 8_193, 8_400):
        b = a.clone()
        b[was] = ((6 + torch.arange(was.numel(), device="cuda") % 2000) << sh) | (b[was] & rest)
        idx = other[torch.randperm(other.numel(), device="cuda")[:held]]
        b[idx] = (5 << sh) | (b[idx] & rest)
        _sort(ctx, b, bits)


@pytest.mark.parametrize("copies", [1, 7, 8, 9, 17, 63, 64, 65, 300])
@pytest.mark.parametrize("bits", [24, 36])
def test_buckets_within_a_bin(ctx, bits, copies):
    """Few distinct values below the top digit, each several times (around the
    fullest bucket that is ordered by comparing, and around the mean that is),
    in all bins and in one of them alone."""
    n = MIN + 4_099
    a = _uniform(n, 8, bits, copies)
    low = bits - 11                                 # 11 top bits, 4,096 keys a bin
    rest = (1 << low) - 1
    few = (a & rest) % max(1, 4096 // copies) * (rest // 4096 + 1)
    _sort(ctx, ((a >> low) << low) | (few & rest), bits)
    b = a.clone()
    one = ((a >> low) == 9).nonzero().flatten()[:copies]
    b[one] = (9 << low) | (b[one] & 1)              # one full bucket, keys out of order
    _sort(ctx, b, bits)


@pytest.mark.parametrize("kb,bits", [(4, 12), (4, 26), (4, 32), (8, 13), (8, 34)])
@pytest.mark.parametrize("n", [(1 << 22) - 1, 1 << 22, (1 << 22) + 16_383])
def test_first_sizes(ctx, kb, bits, n):
    """Around the first size of the top-digit-first form, even keys, one key, and
    few values with the top bits unused."""
    a = _uniform(n, kb, bits, n + bits)
    _sort(ctx, a, bits)
    _sort(ctx, a[:1].repeat(n), bits)
    _sort(ctx, a & ((1 << (bits - 6)) - 1), bits)


@pytest.mark.parametrize("kb", [4, 8])
def test_needs_no_larger_budget_than_the_passes(kb):
    from paper_2607_17571_gb300 import wg

    def least(n):
        """The smallest budget, in units of 256 bytes, that sorts n keys."""
        a = _uniform(n, kb, 8 * kb - 2, n)
        lo, hi = 16, n * kb * 2 // 256
        while lo < hi:
            mid = (lo + hi) // 2
            with wg.Context(0, mem_budget=mid * 256) as c:
                t = a.clone()
                torch.cuda.synchronize()
                try:
                    c.sort_keys(t.data_ptr(), n, kb, 8 * kb - 2)
                    assert torch.equal(t, a.sort().values)
                    hi = mid
                except wg.WgError as e:
                    assert "BUDGET" in str(e)
                    lo = mid + 1
        return lo

    assert least(1 << 22) == least((1 << 22) - 1)  # the first takes the counts if it can


@pytest.mark.parametrize("bits", [6, 13, 18, 34, 62, 64])
@pytest.mark.parametrize("n", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1, 200_003, (1 << 19) + 5])
def test_first_sizes_of_64_bit_keys(ctx, bits, n):
    """Few bins: fewer than the sample's, than a CTA's threads, than CTAs."""
    a = _uniform(n, 8, bits, n + bits)
    _sort(ctx, a, bits)
    _sort(ctx, a[:1].repeat(n), bits)
    _sort(ctx, a & ((1 << (bits - 4)) - 1) if bits < 64 else a >> 1, bits)
