"""Batches at the extremes of their string tables: long runs of empty strings,
strings of a few symbols.

Results against the host preparation and the oracle, bit-exact.  Times are
compared within one run with the same symbols in an ordinary table, so that
no thread may walk a long stretch of the table by itself.
"""
import time

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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _off(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


def _ms(f, reps=7):
    """Least time of a call, in ms (after two warm-up calls)."""
    best = float("inf")
    for i in range(reps + 2):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        if i >= 2:
            best = min(best, (time.perf_counter() - t0) * 1e3)
    return best


@pytest.mark.parametrize("lens", [(5, *(0,) * 3, 6), (5, *(0,) * 4, 6), (5, *(0,) * 5, 6), (1, *(0,) * 4000, 2, 0, 3),
                                  (*(0,) * 9, 2047, *(0,) * 700, 2, *(0,) * 5, 4096, *(0,) * 9)])
def test_build_over_runs_of_empty_strings(ctx, lens):
    off = _off(lens)
    text = np.random.default_rng(len(lens)).integers(0, 3, int(off[-1])).astype(np.uint8)
    got = ctx.build_arrays_batch(_dev(off), _dev(text))
    for a, b in zip(got, W.prep_many(text, off)):
        assert np.array_equal(a.cpu().numpy(), b)


def test_build_time_over_a_run_of_empty_strings(ctx):
    """2^18 empty strings between two others: one thread's walk over them takes 2^18 dependent reads, 5 ms at 20 ns
    each; the two strings alone build in about 0.4 ms."""
    text = _dev(W.dna_iid(100_001, 1))
    plain, empties = _off((50_001, 50_000)), _off((50_001, *(0,) * (1 << 18), 50_000))
    t0 = _ms(lambda: ctx.build_arrays_batch(_dev(plain), text))
    t1 = _ms(lambda: ctx.build_arrays_batch(_dev(empties), text))
    assert t1 < 8 * t0, (t0, t1)


def _outs(n, cap):
    return (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"),
            torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(cap, dtype=torch.int32, device="cuda"))


def _query(ctx, off, lcp, out, **arrays):
    import paper_1501_06663_gb300 as lr
    return lr.lr_batch_query_all(ctx.handle, lr.batch_desc(off, lcp, **arrays), *out)


@pytest.mark.parametrize("front", ["sa", "rank"])
@pytest.mark.parametrize("at", [0, 255, 2 ** 17, 399_998])
def test_a_wrong_offset_anywhere_in_a_long_table(ctx, front, at):
    """400 000 strings of 1 or 2 symbols; one offset is larger than the next."""
    import paper_1501_06663_gb300 as lr
    lens = np.random.default_rng(at).integers(1, 3, 400_000)
    off = _off(lens)
    n = int(off[-1])
    text = np.random.default_rng(at + 1).integers(0, 4, n).astype(np.uint8)
    sa, rank, lcp = ctx.build_arrays_batch(_dev(off), _dev(text))
    out = _outs(n, 4 * n)
    arrays = {"sa": sa} if front == "sa" else {"rank": rank}
    status, total = _query(ctx, _dev(off), lcp, out, **arrays)
    assert status == lr.LR_OK and total >= 0
    wrong = off.copy()
    wrong[at + 1] = off[at + 2] + 1 if at + 2 < off.size - 1 else off[at] - 1
    assert _query(ctx, _dev(wrong), lcp, out, **arrays)[0] == lr.LR_ERR_SENTINEL


@pytest.mark.parametrize("front", ["sa", "rank"])
def test_query_time_of_very_short_strings(ctx, front):
    """4.5 M strings of one symbol against 2197 of 2048: the check of the string table is 36 MB of reads, so the calls
    take about as long as each other (a thread per 2048 symbols checking it: 7 and 20 times as long)."""
    ms = []
    for each in (2048, 1):
        num = 4_500_000 // each
        off = _dev(_off(np.full(num, each)))
        n = num * each
        text = _dev(W.dna_iid(n, 5))
        sa, rank, lcp = ctx.build_arrays_batch(off, text)
        out = _outs(n, 4 * n)
        arrays = {"sa": sa} if front == "sa" else {"rank": rank}
        ms.append(_ms(lambda: _query(ctx, off, lcp, out, **arrays)))
    assert ms[1] < 3 * ms[0], ms


@pytest.mark.parametrize("most", [1, 2, 9, 60, 700, 3000])
def test_short_strings_by_rank(ctx, most):
    """Tiles across strings, a last tile of a few positions: by rank as by sa; ranks out of their string's range and lcp
    sentinels are reported."""
    import paper_1501_06663_gb300 as lr
    rng = np.random.default_rng(most)
    lens = rng.integers(1, most + 1, 120_000 // (most + 1))
    if most > 1:
        lens[::10] = 0                                                     # (a batch has at most n + 1 strings)
    off = _off(lens)
    n = int(off[-1])
    sa, rank, lcp = ctx.build_arrays_batch(_dev(off), _dev(rng.integers(0, 3, n).astype(np.uint8)))
    off = _dev(off)
    want, out = _outs(n, 4 * n), _outs(n, 4 * n)
    st, total = _query(ctx, off, lcp, want, sa=sa)
    assert st == lr.LR_OK and _query(ctx, off, lcp, out, rank=rank) == (st, total)
    assert all(torch.equal(a[:m], b[:m]) for a, b, m in zip(out, want, (n, n, n + 1, total)))
    for at in (0, n // 2, n - 1):
        bad = rank.clone()
        bad[at] = most
        assert _query(ctx, off, lcp, out, rank=bad)[0] == lr.LR_ERR_SENTINEL
        j = int(torch.searchsorted(off, at, right=True)) - 1
        for where in (int(off[j]) + j, int(off[j + 1]) + j):               # its string's first and last lcp entries
            bad = lcp.clone()
            bad[where] = 1
            assert _query(ctx, off, bad, out, rank=rank)[0] == lr.LR_ERR_SENTINEL
