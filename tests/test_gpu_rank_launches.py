"""Queries by rank alone of one string below 2^24 positions: launches and results.

The gather clears what the kernels after it need clear, so one string takes
no launch for that, whichever call came before.  Bit-exact against the oracle.
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1501_06663_gb300 as lrmod
    lrmod.build_library()
    return lrmod


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _arrays(n, seed=1):
    text = W.dna_iid(n, seed)
    m = min(n // 3, 2000)
    text[n - m:] = text[:m]
    sa, rank, lcp = W.prep(text)
    return rank, lcp, oracle.lr_all_raw(rank, lcp)


def _same(got, want):
    return all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(got, want))


def _out(n):
    return (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
            torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(8 * n, dtype=torch.int32, device="cuda"))


def test_launches(lib):
    """Gather, compaction, cover; the walk statistics: gather, compaction, raw lengths, statistics."""
    rank, lcp, want = _arrays(20_000)
    ctx = lib.Context(0)
    try:
        assert _same(ctx.query_all(_dev(lcp), rank=_dev(rank)), want)
        assert lib.lr_last_launch_count(ctx.handle) == 3
        ctx.walk_stats(_dev(lcp), _dev(rank))
        assert lib.lr_last_launch_count(ctx.handle) == 4
    finally:
        ctx.close()


def test_after_calls_of_other_sizes_and_kinds(lib):
    """Status words and tickets left by other calls on the same scratch do not reach a query by rank."""
    small, mid, large = _arrays(8193, 2), _arrays(40_000, 3), _arrays(300_001, 4)
    ctx = lib.Context(0)
    try:
        for rank, lcp, want in (large, small, mid, large, mid):
            r, l = _dev(rank), _dev(lcp)
            assert _same(ctx.query_all(l, rank=r), want)
            start, length = ctx.query_leftmost(l, rank=r)
            assert _same((length, start), want)
            assert _same(ctx.query_all_raw(l, r), want)
            assert _same(ctx.query_all(l, rank=r), want)
            stats, (alpha, beta) = ctx.walk_stats(l, r), oracle.walk_counts(rank, lcp)[:2]
            assert (stats["alpha_sum"], stats["beta_sum"]) == (int(alpha.sum()), int(beta.sum()))
            assert (stats["alpha_max"], stats["beta_min"]) == (int(alpha.max()), int(beta.min()))
            assert _same(ctx.query_all(l, rank=r), want)
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1, 2, 2047, 2048, 2049, 8191, 8192, 8193, 16_385, 100_003])
def test_static(lib, n):
    rank, lcp, want = _arrays(n, n)
    out = _out(n)
    for _ in range(2):
        status, total = lib.lr_query_all_static(_dev(rank), _dev(lcp), *out)
        assert status == lib.LR_OK and total == want[3].size
        assert _same((*out[:3], out[3][:total]), want)
    bad = rank.copy()
    bad[n // 2] = n
    assert lib.lr_query_all_static(_dev(bad), _dev(lcp), *out)[0] == lib.LR_ERR_SENTINEL
    status, total = lib.lr_query_all_static(_dev(rank), _dev(lcp), *out)
    assert status == lib.LR_OK and _same((*out[:3], out[3][:total]), want)
