"""Which path a query takes by its size: one tile, the dense array, the partition.

Strings of at most 8192 positions take one launch; up to a few million
positions (2^24 are more, in a batch too) the lengths go through a dense
array; above, through the radix partition.  Each path at the edges of its range and with wrong inputs, against
the oracle, or at large sizes against the gather front end.  Integers:
bit-exact.
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = None


@pytest.fixture(scope="module")
def ctx():
    global P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1501_06663_gb300 as lrmod
    lrmod.build_library()
    P = lrmod
    c = lrmod.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _text(kind, n):
    rng = np.random.default_rng(n)
    if kind == "one":
        return np.full(n, 97, np.uint8)
    if kind == "bytes":
        return rng.integers(0, 256, n).astype(np.uint8)
    if kind == "copy":                                     # the second half repeats the first
        h = rng.integers(65, 69, (n + 1) // 2).astype(np.uint8)
        return np.concatenate([h, h])[:n]
    return W.make_text(kind, n, n)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 256, 2047, 2049, 4099, 8191, 8192, 8193, 20001])
@pytest.mark.parametrize("kind", ["one", "bytes", "copy", "protein", "english"])
def test_every_size_of_short_strings(ctx, kind, n):
    text = _text(kind, n)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    L = np.maximum(lcp[rank], lcp[rank + 1])
    m = int(((L > 0) & (L >= np.concatenate([[0], L[:-1]]))).sum())
    for kw in ({"sa": _dev(sa)}, {"rank": _dev(rank)}):
        got = ctx.query_all(_dev(lcp), **kw)
        for a, b in zip(got, want):
            assert np.array_equal(a.cpu().numpy(), b)
        assert P.lr_last_compact_size(ctx.handle) == m
        st, ln = ctx.query_leftmost(_dev(lcp), **kw)
        assert np.array_equal(st.cpu().numpy(), want[1]) and np.array_equal(ln.cpu().numpy(), want[0])


def _wrong(sa, rank, lcp, n):
    i = n // 2
    for what in ("sa twice", "sa past", "sa negative", "rank past", "lcp first", "lcp last", "lcp long", "lcp negative"):
        a, r, l = sa.clone(), rank.clone(), lcp.clone()
        if what == "sa twice":
            a[i] = a[i + 1]
        elif what == "sa past":
            a[i] = n
        elif what == "sa negative":
            a[i] = -1
        elif what == "rank past":
            r[i] = n
        elif what == "lcp first":
            l[0] = 1
        elif what == "lcp last":
            l[n] = 1
        elif what == "lcp long":
            l[i] = n
        else:
            l[i] = l[i + 1] = -2
        if what != "rank past":
            yield what, {"sa": a}, l
        if not what.startswith("sa"):
            yield what, {"rank": r}, l


@pytest.mark.parametrize("n", [3000, 8192, 8193, 100_000, (1 << 20) + 1])
def test_wrong_inputs_are_reported(ctx, n):
    text = torch.from_numpy(W.dna_iid(n, 5)).cuda()
    sa, rank, lcp = ctx.build_arrays(text)
    want = ctx.query_all(lcp, rank=rank)
    for what, kw, bad in _wrong(sa, rank, lcp, n):
        with pytest.raises(P.LRError) as e:
            ctx.query_all(bad, **kw)
        assert e.value.status == P.LR_ERR_SENTINEL, (what, kw.keys())
        with pytest.raises(P.LRError) as e:
            ctx.query_leftmost(bad, **kw)
        assert e.value.status == P.LR_ERR_SENTINEL, (what, kw.keys())
    for kw in ({"sa": sa}, {"rank": rank}):                # the context stays usable
        for a, b in zip(ctx.query_all(lcp, **kw), want):
            assert torch.equal(a, b)


def test_capacity_in_one_tile(ctx):
    text = W.make_text("protein", 4000, 3)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    n = text.size
    out = [torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
           torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.full((1003,), -7, dtype=torch.int32, device="cuda")]
    st, total = P.lr_query_all(ctx.handle, _dev(sa), None, _dev(lcp), out[0], out[1], out[2], out[3][:1000])
    assert st == P.LR_ERR_CAPACITY and total == want[3].size
    assert np.array_equal(out[2].cpu().numpy(), want[2]) and np.array_equal(out[0].cpu().numpy(), want[0])
    assert np.array_equal(out[3].cpu().numpy(), np.concatenate([want[3][:1000], [-7] * 3]))


@pytest.fixture(scope="module")
def large_batch(ctx):
    """More than 2^24 positions: thousands of tiny strings, strings on and next to round edges, two long ones."""
    rng = np.random.default_rng(8)
    lens = np.concatenate([rng.integers(0, 9, 9000), [8192, 5 * 4096 + 100, 4096, 1], rng.integers(3000, 9000, 40),
                           [9_000_001, 0, 7_700_000, 5]])
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    assert off[-1] > 1 << 24
    text = rng.integers(0, 3, int(off[-1])).astype(np.uint8)
    text[-3_000_000:-2_990_000] = text[-6_000_000:-5_990_000]   # lengths that escape their fields
    d_off, d_text = _dev(off), _dev(text)
    return off, d_off, ctx.build_arrays_batch(d_off, d_text)


def test_large_batch_against_the_gather(ctx, large_batch):
    _, off, (sa, rank, lcp) = large_batch
    want = ctx.query_batch(off, lcp, rank=rank)
    for a, b in zip(ctx.query_batch(off, lcp, sa=sa), want):
        assert torch.equal(a, b)


def test_wrong_large_batch_is_reported(ctx, large_batch):
    h_off, off, (sa, rank, lcp) = large_batch
    num, n = off.numel() - 1, int(h_off[-1])
    out = [torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
           torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(6 * n, dtype=torch.int32, device="cuda")]
    big = num - 4                                          # the string of 9 000 001 positions
    at = int(h_off[big])
    for what in ("twice", "past", "first sentinel", "last sentinel", "offsets"):
        a, l, o = sa.clone(), lcp.clone(), off.clone()
        if what == "twice":
            a[at + 5000] = a[at + 5001]
        elif what == "past":
            a[at + 5000] = 9_000_001
        elif what == "first sentinel":
            l[at + big] = 1
        elif what == "last sentinel":
            l[at + big + 9_000_001] = 1
        else:
            o[big] = o[big + 1] + 7
        st, _ = P.lr_batch_query_all(ctx.handle, P.batch_desc(o, l, sa=a), *out)
        assert st == P.LR_ERR_SENTINEL, what
    st, total = P.lr_batch_query_all(ctx.handle, P.batch_desc(off, lcp, sa=sa), *out)
    assert st == P.LR_OK and total == int(out[2][n])


@pytest.mark.parametrize("n", [5000, 300_000, 5_500_000, (1 << 24) + 77])
@pytest.mark.parametrize("front", ["sa", "rank"])
def test_alternating_inputs_without_waiting(ctx, n, front):
    """Queries of two inputs in turn on one context and one stream: no kernel sees what an earlier query left."""
    sets = []
    for seed in (1, 2):
        text = torch.from_numpy(W.dna_iid(n, seed)).cuda()
        sa, rank, lcp = ctx.build_arrays(text)
        off = torch.tensor([0, n], dtype=torch.int64, device="cuda")
        want = ctx.query_batch(off, lcp, rank=rank) if front == "sa" else ctx.query_batch(off, lcp, sa=sa)
        kw = {"sa": sa, "rank": None} if front == "sa" else {"sa": None, "rank": rank}
        sets.append((kw, lcp, [t.clone() for t in want]))
    rounds = 12
    outs = [(torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
             torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(3 * n, dtype=torch.int32, device="cuda"))
            for _ in range(rounds)]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        kw, lcp, _ = sets[i % 2]
        st, _ = P.lr_query_all(ctx.handle, kw["sa"], kw["rank"], lcp, *out, sync=False)
        assert st == P.LR_OK
    assert P.lr_device_status(ctx.handle) == P.LR_OK
    for i, out in enumerate(outs):
        want = sets[i % 2][2]
        for a, b in zip(out[:3], want):
            assert torch.equal(a, b)
        assert torch.equal(out[3][:want[3].numel()], want[3])
