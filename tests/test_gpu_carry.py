"""The cover kernel's switch between the staged carry and the walk in place.

The entries that reach a tile from before it are staged up to 64; the kernel
takes the other path when all 64 staged ones reach the tile and more entries
precede them.  Texts in which exactly 63, 64 or 65 compact repeats reach a
tile's first position, as its only predecessors or after others.
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _text(carry, edge, first, grow):
    """Repeats of R start at `carry` consecutive positions before `edge` and end past it, at the text's start (first) or
    after random letters; equally long, or (grow) each one symbol longer than the one before."""
    rng = np.random.default_rng(carry + 1000 * grow)
    at = 0 if first else edge - 2 * carry
    length = edge + 9 if first else 3 * carry
    R = rng.integers(0, 100, 2 * carry + length).astype(np.uint8)
    parts = [rng.integers(0, 100, at).astype(np.uint8), R]
    for j in range(carry):
        parts += [R[j:j + length + grow * j], rng.integers(100, 256, 4).astype(np.uint8)]
    parts.append(rng.integers(0, 100, 20_000).astype(np.uint8))
    return np.concatenate(parts)


@pytest.mark.parametrize("code,edge,first", [(8, 2048, True), (8, 2048, False), (8, 8192, False), (9, 4096, True),
                                             (9, 8192, False), (12, 8192, True), (12, 8192, False)])
@pytest.mark.parametrize("grow", [0, 1])
@pytest.mark.parametrize("carry", [63, 64, 65, 66, 130])
def test_carry(tmp_path, carry, code, edge, first, grow):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1501_06663_gb300 as lr
    lr.build_library()
    text = _text(carry, edge, first, grow)
    sa, rank, lcp = W.prep(text)
    start, length = oracle.compact(rank, lcp)
    reach = (start < edge) & (start + length > edge)
    assert int(reach.sum()) == carry and (int((start < edge).sum()) > carry) == (not first)
    want = oracle.lr_all_compact(rank, lcp)
    (tmp_path / "codes").write_text("".join("%d %d\n" % (a * 64 + b, code) for a in range(32) for b in range(32)))
    ctx = lr.Context(0)
    try:
        lr.lr_autotune_load(ctx.handle, str(tmp_path / "codes"))
        dsa, dlcp = torch.from_numpy(sa).cuda(), torch.from_numpy(lcp).cuda()
        for a, b in zip(ctx.query_all(dlcp, sa=dsa), want):
            assert np.array_equal(a.cpu().numpy(), b)
        st, ln = ctx.query_leftmost(dlcp, sa=dsa)
        assert np.array_equal(st.cpu().numpy(), want[1]) and np.array_equal(ln.cpu().numpy(), want[0])
    finally:
        ctx.close()
