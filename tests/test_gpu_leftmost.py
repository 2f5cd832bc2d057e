"""The leftmost query where many compact left-bounded repeats overlap.

Results against the oracle (small) and against the all-repeats query (large),
bit-exact; the time of the tile cover against the warp-segment cover on the
same arrays.
"""
import statistics

import numpy as np
import pytest

import oracle
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


def _shift_register(k, t, n):
    """x[i + k] = x[i + t] ^ x[i], a primitive recurrence: every word of k - 1 symbols but the zero one occurs twice, so
    a repeat of k - 1 symbols starts at every position."""
    x = [1] * k
    for i in range(n - k):
        x.append(x[i] ^ x[i + t])
    return np.array(x, np.uint8)


def _text(kind, n):
    rng = np.random.default_rng(n)
    if kind == "ties":
        return _shift_register(*{32767: (15, 1), 131071: (17, 3)}[n], n)
    if kind == "binary":
        return rng.integers(0, 2, n).astype(np.uint8)
    if kind == "tandem":                                   # repeats that shrink towards each change
        text = np.resize(rng.integers(0, 4, 97), n)
        text[rng.integers(0, n, n // 300)] ^= 1
        return text.astype(np.uint8)
    a = rng.integers(0, 4, n // 2)                         # a text and its copy with single changes
    b = a.copy()
    b[rng.integers(0, a.size, a.size // 100)] ^= 1
    return np.concatenate([a, b]).astype(np.uint8)


def _with_code(code, path):
    import paper_1501_06663_gb300 as lr
    c = lr.Context(0)
    path.write_text("".join("%d %d\n" % (a * 64 + b, code) for a in range(32) for b in range(32)))
    lr.lr_autotune_load(c.handle, str(path))
    return c


CASES = [("binary", 3000), ("binary", 8192), ("binary", 8193), ("binary", 70_001), ("tandem", 8000), ("tandem", 50_000),
         ("copy", 6000), ("copy", 40_000)]


@pytest.mark.parametrize("code", [8, 9, 12])
@pytest.mark.parametrize("kind,n", CASES)
def test_against_the_oracle(tmp_path, kind, n, code):
    text = _text(kind, n)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    c = _with_code(code, tmp_path / "codes")
    try:
        for arrays in ({"sa": _dev(sa)}, {"rank": _dev(rank)}):
            start, length = c.query_leftmost(_dev(lcp), **arrays)
            assert np.array_equal(length.cpu().numpy(), want[0]) and np.array_equal(start.cpu().numpy(), want[1])
    finally:
        c.close()


@pytest.mark.parametrize("n", [32767, 131071])
def test_ties_everywhere(ctx, n):
    text = _text("ties", n)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    start, length = ctx.query_leftmost(_dev(lcp), sa=_dev(sa))
    assert np.array_equal(length.cpu().numpy(), want[0]) and np.array_equal(start.cpu().numpy(), want[1])


@pytest.mark.parametrize("n", [(1 << 23) + 777])
def test_large_against_the_all_query(ctx, n):
    text = _dev(_text("binary", n))
    sa, rank, lcp = ctx.build_arrays(text)
    want = ctx.query_all(lcp, sa=sa)
    start, length = ctx.query_leftmost(lcp, sa=sa)
    assert torch.equal(length, want[0]) and torch.equal(start, want[1])


@pytest.mark.parametrize("kind", ["ties", "binary"])
def test_time_against_the_warp_segments(tmp_path, kind):
    """Where 22 repeats of one length (or binary text's 20) cover a position, the tile cover's scans must not make it
    much slower than the warp-segment cover, whose cost depends less on the overlap (2.2 and 1.4 times as long while
    the scans also counted the ties)."""
    import paper_1501_06663_gb300 as lr
    n = (1 << 23) - 1 if kind == "ties" else 1 << 25
    if kind == "ties":
        x = torch.from_numpy(_shift_register(23, 5, 400).astype(np.uint8)).cuda()
        j = 0                                              # squares of the recurrence: longer and longer steps
        while x.numel() < n:
            while 23 << (j + 1) <= x.numel():
                j += 1
            k, t, size = 23 << j, 5 << j, x.numel()
            x = torch.cat([x, x[size - k:size - t] ^ x[size - k + t:size]])
        text = x[:n].contiguous()
    else:
        text = _dev(_text(kind, n))
    builder = lr.Context(0)
    sa, rank, lcp = builder.build_arrays(text)
    builder.close()
    ms, got = [], []
    for code in (0, 8):
        c = _with_code(code, tmp_path / "codes")
        lr.lr_set_phase_timing(c.handle, True)
        cover = []
        for i in range(9):
            got.append(c.query_leftmost(lcp, sa=sa))
            if i >= 2:
                cover.append(lr.lr_phase_times(c.handle)[-1])
        ms.append(statistics.median(cover))
        c.close()
    assert all(torch.equal(a, b) for g in got for a, b in zip(g, got[0]))
    assert ms[1] < 1.25 * ms[0], ms

