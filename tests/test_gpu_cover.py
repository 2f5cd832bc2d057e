"""The cover kernel where its links between equal entries and its carry go past their short forms.

Position k's holders are linked by distances of one byte; a text is built in
which the next compact LLR of the same length lies 253 .. 400 entries further
on (shorter ones between), and the number of entries over a tile's first
position passes the 64 that are staged.  Integers: bit-exact.
"""
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


def _far_text(between, length, lead):
    """A random stretch R with copies of R[lead : +length], of every second
    R[lead + 2j : +length - 1] (1 <= j <= between) and of
    R[lead + 2 (between + 1) : +length]: the first and the last are equal, the
    ones between shorter."""
    rng = np.random.default_rng(between * 1009 + lead)
    end = lead + 2 * (between + 1)
    R = rng.integers(0, 200, end + length + 5).astype(np.uint8)
    parts = [R]
    for j in range(between + 2):
        a = lead + 2 * j
        ln = length if j in (0, between + 1) else length - 1
        parts += [R[a:a + ln], rng.integers(200, 256, 3).astype(np.uint8)]
    return np.concatenate(parts)


@pytest.mark.parametrize("between,length,lead", [(30, 100, 2000), (62, 200, 2040), (64, 200, 2050), (253, 700, 100),
                                                 (254, 700, 100), (255, 700, 100), (400, 900, 3), (400, 900, 1700)])
def test_equal_entries_far_apart(ctx, between, length, lead):
    text = _far_text(between, length, lead)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    k = lead + 2 * (between + 1)                       # covered by the first and the last copy
    assert want[0][k] == length and want[2][k + 1] - want[2][k] == 2
    dsa, dlcp = torch.from_numpy(sa).cuda(), torch.from_numpy(lcp).cuda()
    got = ctx.query_all(dlcp, sa=dsa)
    for a, b in zip(got, want):
        assert np.array_equal(a.cpu().numpy(), b)
    st, ln = ctx.query_leftmost(dlcp, sa=dsa)
    assert np.array_equal(st.cpu().numpy(), want[1]) and np.array_equal(ln.cpu().numpy(), want[0])


def _tied_text(width, blocks):
    """Blocks in which up to `width` + 1 equal repeats cover a position: R and all its windows of width + 1."""
    rng = np.random.default_rng(width)
    parts = []
    for _ in range(blocks):
        R = rng.integers(0, 200, 2 * width + 2).astype(np.uint8)
        parts.append(R)
        for j in range(width):
            parts += [R[j:j + width + 1], rng.integers(200, 256, 2).astype(np.uint8)]
    return np.concatenate(parts)


@pytest.mark.parametrize("width,blocks", [(3, 1200), (13, 130), (14, 130), (15, 130), (16, 130), (40, 20)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_tie_counts_and_unaligned_offsets(ctx, width, blocks, shift):
    """Counts around the 15 that the byte prefixes take; offsets[] 8, 16 or 24 bytes off a 32-byte boundary."""
    import paper_1501_06663_gb300 as lrmod
    text = _tied_text(width, blocks)
    sa, rank, lcp = W.prep(text)
    want = oracle.lr_all_raw(rank, lcp)
    assert int(np.diff(want[2]).max()) >= width
    n = text.size
    ln, st = (torch.empty(n + shift, dtype=torch.int32, device="cuda")[shift:] for _ in range(2))
    off = torch.empty(n + 1 + shift, dtype=torch.int64, device="cuda")[shift:]
    starts = torch.full((want[3].size + 1 + shift,), -7, dtype=torch.int32, device="cuda")[shift:]
    status, total = lrmod.lr_query_all(ctx.handle, torch.from_numpy(sa).cuda(), None, torch.from_numpy(lcp).cuda(), ln, st,
                                       off, starts[:-1])
    assert status == lrmod.LR_OK and total == want[3].size
    for a, b in zip((ln, st, off, starts[:-1]), want):
        assert np.array_equal(a.cpu().numpy(), b)
    assert int(starts[-1]) == -7
