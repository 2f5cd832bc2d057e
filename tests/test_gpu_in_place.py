"""Outputs that replace the inputs: lr_len in the lcp array, lr_start in sa or rank.

Every call writes its outputs after all inputs have been read, on each path,
with repeats longer than the 2-byte and 12-bit length fields hold (65534 and
4095).  Against the same query out of place.
"""
import pytest

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


def _arrays(ctx, n):
    """A text that repeats its first half."""
    text = torch.from_numpy(W.dna_iid(n, n)).cuda()
    text[n - n // 2:] = text[:n // 2].clone()
    return ctx.build_arrays(text)


@pytest.mark.parametrize("n", [1000, 8192, 8193, 150_001, 1 << 20, (5 << 20) + 1, 1 << 24])
@pytest.mark.parametrize("call", ["sa", "rank", "static", "batch"])
def test_in_place(lib, n, call):
    if call == "static" and n > lib.LR_STATIC_MAX_N:
        pytest.skip("beyond the static call")
    ctx = lib.Context(0)
    try:
        sa, rank, lcp = _arrays(ctx, n)
        assert n < 150_000 or int(lcp.max()) > 65534
        want = ctx.query_all(lcp, sa=sa)
        front = sa if call in ("sa", "batch") else rank
        ln, st = lcp[:n], front                            # the first n words of lcp, and sa or rank
        off = torch.empty(n + 1, dtype=torch.int64, device="cuda")
        starts = torch.empty(int(want[3].numel()), dtype=torch.int32, device="cuda")
        if call == "static":
            status, total = lib.lr_query_all_static(rank, lcp, ln, st, off, starts)
        elif call == "batch":
            table = torch.tensor([0, n], device="cuda")
            status, total = lib.lr_batch_query_all(ctx.handle, lib.batch_desc(table, lcp, sa=sa), ln, st, off, starts)
        else:
            status, total = lib.lr_query_all(ctx.handle, sa if call == "sa" else None, rank if call == "rank" else None, lcp,
                                             ln, st, off, starts)
        assert status == lib.LR_OK
        for a, b in zip((ln, st, off, starts), want):
            assert torch.equal(a, b)
    finally:
        ctx.close()
