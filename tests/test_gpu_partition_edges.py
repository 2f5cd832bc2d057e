"""The radix partition by sa at the edges of its rounds, buckets and super-buckets.

One string above 5 * 2^20 positions, batches above 12 * 2^20 (below, the
lengths go to a dense array): sizes with a last round, bucket or super-bucket
of one position, full ones and ones short of one, and both sides of the line.
Against the gather by rank, bit-exact; wrong inputs are reported.
"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MI = 1 << 20
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


def _same(got, want):
    return all(torch.equal(a, b) for a, b in zip(got, want))


def _text(n, seed):
    """DNA with a repeat of over 4095 symbols (its length escapes the 12-bit field) that ends at the last position."""
    text = W.dna_iid(n, seed)
    text[n - 5000:] = text[:5000]
    return torch.from_numpy(text).cuda()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [5 * MI, 5 * MI + 1, 6 * MI - 1, 6 * MI, 6 * MI + 1, 6 * MI + 4095, 6 * MI + 4096, 6 * MI + 4097,
                               6 * MI + 32767, 6 * MI + 32768, 6 * MI + 32769, 7 * MI - 32767, 7 * MI - 4095])
def test_one_string(ctx, n, shift):
    """shift = 1: arrays that start 4 bytes past a 16-byte boundary (no bulk copies)."""
    sa, rank, lcp = ctx.build_arrays(_text(n, n))
    want = ctx.query_batch(torch.tensor([0, n], device="cuda"), lcp, rank=rank)
    if shift:
        sa, lcp = torch.cat([sa[:1], sa])[1:], torch.cat([lcp[:1], lcp])[1:]
        assert sa.data_ptr() % 16 and lcp.data_ptr() % 16
    assert _same(ctx.query_all(lcp, sa=sa), want)
    start, length = ctx.query_leftmost(lcp, sa=sa)
    assert _same((length, start), want)


def _batch(ctx, lens, seed):
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)).cuda()
    n = int(off[-1])
    return off, n, ctx.build_arrays_batch(off, _text(n, seed))


@pytest.mark.parametrize("lens", [
    (12 * MI,), (12 * MI + 1,), (13 * MI + 1,),                                   # both sides of the line
    (1, 4096 * 3, 0, 0, 4095, 4097, 32768, 5 * MI, 1, 8 * MI - 3, 2),
    (4096,) * 3100 + (1,), (4095,) * 3100, (4097,) * 3100,                        # rounds inside and across strings
    (300_007,) * 43, (3,) * 300_000 + (12 * MI,)])
def test_batches(ctx, lens):
    off, n, (sa, rank, lcp) = _batch(ctx, lens, len(lens))
    want = ctx.query_batch(off, lcp, rank=rank)
    assert _same(ctx.query_batch(off, lcp, sa=sa), want)


def test_broken_sentinels_of_a_batch(ctx):
    """The first lcp entry of a string that starts on a round and fills whole rounds, the last entry of the string before
    and of one that ends inside a round."""
    lens = (8192, 5 * 4096 + 100, 3000, 12 * MI, 4096)
    off, n, (sa, rank, lcp) = _batch(ctx, lens, 3)
    want = ctx.query_batch(off, lcp, rank=rank)
    out = (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
           torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(4 * n, dtype=torch.int32, device="cuda"))
    first = [int(off[j]) + j for j in range(5)]                                   # of each string's lcp entries
    for where in (0, first[1] - 1, first[1], first[2] - 1, first[3], first[4] - 1, first[4], n + 4):
        bad = lcp.clone()
        bad[where] = 5
        assert P.lr_batch_query_all(ctx.handle, P.batch_desc(off, bad, sa=sa), *out)[0] == P.LR_ERR_SENTINEL, where
    assert _same(ctx.query_batch(off, lcp, sa=sa), want)


@pytest.mark.parametrize("n", [6 * MI + 70_000, 6 * MI])
@pytest.mark.parametrize("what", ["twice near", "twice far", "negative", "past the end", "long lcp", "negative lcp", "sentinel"])
def test_wrong_input_is_reported(ctx, n, what):
    sa, rank, lcp = ctx.build_arrays(_text(n, 11))
    bad_sa, bad_lcp = sa.clone(), lcp.clone()
    if what == "twice near":                                                      # in one bucket of 2^15
        r = torch.nonzero((sa >> 15) == (sa[5000] >> 15)).reshape(-1)
        bad_sa[5000] = sa[r[r != 5000][7]]
    elif what == "twice far":
        bad_sa[4097] = 0 if int(sa[4097]) != 0 else n - 1
    elif what == "negative":
        bad_sa[9000] = -5
    elif what == "past the end":
        bad_sa[9000] = n
    elif what == "long lcp":
        bad_lcp[9000] = n
    elif what == "negative lcp":
        bad_lcp[9000] = bad_lcp[9001] = -3
    else:
        bad_lcp[n] = 1
    with pytest.raises(P.LRError) as e:
        ctx.query_all(bad_lcp, sa=bad_sa)
    assert e.value.status == P.LR_ERR_SENTINEL
    assert _same(ctx.query_all(lcp, sa=sa), ctx.query_batch(torch.tensor([0, n], device="cuda"), lcp, rank=rank))
