"""The GPU array build where its tiles, groups and keys have their edges.

Tiles of 2048 positions (keys) and of 2048 sorted suffixes (groups that run
over many tiles), alphabets from one symbol (63 per round-0 key) to all 256
byte values, strings shorter than a key.  Against the host preparation,
bit-exact.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1501_06663_gb300 as lrmod
    lrmod.build_library()
    c = lrmod.Context(0)
    yield c
    c.close()


def _text(kind, n):
    rng = np.random.default_rng(n)
    if kind == "one":
        return np.full(n, 97, np.uint8)
    if kind == "period2":
        return np.resize(np.frombuffer(b"ab", np.uint8), n).copy()
    if kind == "blocks":                               # long runs: groups over many tiles in every round
        return np.repeat(rng.integers(0, 3, n // 700 + 1), 700)[:n].astype(np.uint8)
    if kind == "bytes":
        return rng.integers(0, 256, n).astype(np.uint8)
    return W.dna_planted(n, n)


@pytest.mark.parametrize("n", [1, 2, 7, 63, 64, 2047, 2048, 2049, 4096 + 62, 30011])
@pytest.mark.parametrize("kind", ["one", "period2", "blocks", "bytes", "dna"])
def test_one_string(ctx, kind, n):
    text = _text(kind, n)
    got = ctx.build_arrays(torch.from_numpy(text).cuda())
    for a, b in zip(got, W.prep(text)):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("lens", [(0, 1, 0, 2, 5), (2048, 2048), (2047, 1, 2049, 0, 3), (5,) * 1500, (4100, 9, 8, 7, 64, 63)])
@pytest.mark.parametrize("kind", ["one", "blocks", "bytes"])
def test_many_strings(ctx, kind, lens):
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    text = _text(kind, int(off[-1]))
    sa, rank, lcp = ctx.build_arrays_batch(torch.from_numpy(off).cuda(), torch.from_numpy(text).cuda())
    wsa, wrank, wlcp = W.prep_many(text, off)
    assert np.array_equal(sa.cpu().numpy(), wsa) and np.array_equal(rank.cpu().numpy(), wrank)
    assert np.array_equal(lcp.cpu().numpy(), wlcp)


@pytest.mark.parametrize("n", [(30 << 20) + 5, (40 << 20) + 3, (13 << 24) + 1])
def test_ranks_back_to_position_order(ctx, n):
    """Round 0's ranks scattered in windows of 2^24 positions (the last one partial), and past 13 windows sorted
    back: the suffix array is a permutation in suffix order."""
    text = torch.from_numpy(W.dna_iid(n, 3)).cuda()
    text[n // 2: n // 2 + 3000] = text[:3000]              # a few more rounds
    sa, rank, lcp = ctx.build_arrays(text)
    assert torch.equal(rank[sa.long()], torch.arange(n, dtype=torch.int32, device="cuda"))
    # sampled neighbours: lcp symbols equal, the next one in order
    r = torch.randint(1, n, (200_000,), device="cuda")
    r[:2] = torch.stack([rank[0], rank[n // 2]]).long().clamp(min=1)
    x, y, m = sa[r - 1].long(), sa[r].long(), lcp[r].long()
    for t in range(int(m.max()) + 1):
        a = torch.where(x + t < n, text[(x + t).clamp(max=n - 1)].long(), -1)
        b = torch.where(y + t < n, text[(y + t).clamp(max=n - 1)].long(), -1)
        assert bool((a[m > t] == b[m > t]).all()) and bool((a[m == t] < b[m == t]).all())
