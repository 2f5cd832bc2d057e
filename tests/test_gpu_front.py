"""The rank-order front end at the edges of its rounds, buckets and super-buckets.

Rounds of 4096 ranks, chunks of 256 and buckets of 2^15 positions,
super-buckets of 2^20: full ones take unchecked paths, partial ones and wrong
inputs the checked ones.  Small sizes against the oracle, large ones against
the gather front end (rank alone, as a one-string batch).  Integers: bit-exact.
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


def _text(n, seed):
    """DNA with a repeat of over 4095 symbols (a length that escapes its field) that ends at the last position."""
    text = W.dna_iid(n, seed)
    m = min(5000, n // 3)
    text[n - m:] = text[:m]
    return text


@pytest.mark.parametrize("n", [255, 4095, 4096, 4097, 8192, 32767, 32768, 32769, 65536 + 256, (1 << 20) - 1, 1 << 20,
                               (1 << 20) + 1, (1 << 20) + 32768])
def test_sizes_at_the_edges(ctx, n):
    text = _text(n, n)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    got = ctx.query_all(_dev(lcp), sa=_dev(sa))
    for a, b in zip(got, want):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("n", [(1 << 24) + (1 << 15), (1 << 24) + 4095, 40_000_003])
@pytest.mark.parametrize("shift", [0, 1])
def test_large_sizes_against_the_gather(ctx, n, shift):
    """shift = 1: arrays that start 4 bytes past a 16-byte boundary (no bulk copies)."""
    text = torch.from_numpy(_text(n, 7)).cuda()
    sa, rank, lcp = ctx.build_arrays(text)
    off = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    want = ctx.query_batch(off, lcp, rank=rank)
    if shift:
        sa = torch.cat([sa[:1], sa])[1:]
        lcp = torch.cat([lcp[:1], lcp])[1:]
        assert sa.data_ptr() % 16 and lcp.data_ptr() % 16
    got = ctx.query_all(lcp, sa=sa)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    st, ln = ctx.query_leftmost(lcp, sa=sa)
    assert torch.equal(ln, want[0]) and torch.equal(st, want[1])


@pytest.mark.parametrize("n", [3 * 32768, 3 * 32768 + 17, (1 << 20) + 40000, (1 << 24) + 70000])
def test_wrong_sa_in_full_rounds_is_reported(ctx, n):
    text = torch.from_numpy(W.dna_iid(n, 11)).cuda()
    sa, _, lcp = ctx.build_arrays(text)
    want = ctx.query_all(lcp, sa=sa)
    for what in ("twice near", "twice far", "negative", "past the end", "long lcp", "negative lcp", "sentinel"):
        bad_sa, bad_lcp = sa.clone(), lcp.clone()
        if what == "twice near":                       # inside one bucket, most likely
            r = int(torch.nonzero((bad_sa >> 15) == (bad_sa[5000] >> 15))[7])
            bad_sa[5000] = bad_sa[r] if r != 5000 else bad_sa[r + 1]
        elif what == "twice far":
            bad_sa[4097] = 0 if int(sa[4097]) != 0 else n - 1
        elif what == "negative":
            bad_sa[9000] = -5
        elif what == "past the end":
            bad_sa[9000] = n
        elif what == "long lcp":
            bad_lcp[9000] = n
        elif what == "negative lcp":
            bad_lcp[9000] = -3
            bad_lcp[9001] = -3
        else:
            bad_lcp[n] = 1
        with pytest.raises(P.LRError) as e:
            ctx.query_all(bad_lcp, sa=bad_sa)
        assert e.value.status == P.LR_ERR_SENTINEL, what
    got = ctx.query_all(lcp, sa=sa)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
