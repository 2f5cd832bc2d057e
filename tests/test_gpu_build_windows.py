"""The array build above 30 * 2^20 positions with many suffixes unsettled for several rounds.

There a round's rank words go to position order in windows of 2^24 positions
(up to 19 of them, from 2^18 unsettled suffixes on) and straight above.  The
arrays are checked against their definition: rank inverts sa, and of sampled
sa neighbours the first lcp symbols are equal and the next ones in order.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MI = 1 << 20


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1501_06663_gb300 as lrmod
    lrmod.build_library()
    c = lrmod.Context(0)
    yield c
    c.close()


def _text(n, every):
    """Four letters, the last quarter a copy of the first with one letter in `every` changed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    text = torch.randint(0, 4, (n,), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    q = n // 4
    text[n - q:] = text[:q]
    at = n - q + torch.randint(0, q, (q // every,), generator=g, device="cuda")
    text[at] = (text[at] + 1) % 4
    return text


@pytest.mark.parametrize("n", [30 * MI, 30 * MI + 5, 40 * MI + 3, (13 << 24) + 1, (19 << 24) + 1])
def test_many_rounds_of_many_suffixes(ctx, n):
    text = _text(n, 200)
    sa, rank, lcp = ctx.build_arrays(text)
    assert torch.equal(rank[sa.long()], torch.arange(n, dtype=torch.int32, device="cuda"))
    # 21 symbols per key, twice as many each round; a suffix is unsettled while a neighbour shares more
    longest = torch.maximum(lcp[:-1], lcp[1:])
    left = [int((longest >= 21 << r).sum()) for r in range(3)]
    assert min(left) > 1 << 18 and any(a % 2048 for a in left), left
    del longest
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    r = torch.randint(1, n, (400_000,), generator=g, device="cuda")
    x, y, m = sa[r - 1].long(), sa[r].long(), lcp[r].long()
    alive = torch.arange(r.numel(), device="cuda")
    t = 0
    while alive.numel():                                   # those whose first t symbols are equal
        a, b = x[alive] + t, y[alive] + t
        ca = torch.where(a < n, text[a.clamp(max=n - 1)].int(), -1)
        cb = torch.where(b < n, text[b.clamp(max=n - 1)].int(), -1)
        ends = m[alive] == t
        assert bool((ca[ends] < cb[ends]).all()) and bool((ca[~ends] == cb[~ends]).all())
        alive = alive[~ends]
        t += 1
