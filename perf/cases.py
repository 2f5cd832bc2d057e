"""What this library does for its users, as cases that can be timed.

A case is one call (or one launch of a captured plan) through the Python
binding, on synthetic text of the kinds the workloads package stands for:
English-like text, DNA (order-2 Markov with planted, mutated repeats, or
i.i.d.), protein with tandem arrays, and batches of such strings.  Texts are
made on the GPU from the seed; their arrays come from the library's own build.

Keys of a case: "op" (all, leftmost, batch, plan, host, build), "kind" of
text, "n" positions, "front" (sa or rank given to the query), and for batches
"count" strings of lengths spread log-uniformly over [lo, hi] or lognormally
around 10^5 (the serving mix).  The lengths depend on the case alone, their
order and the text on the seed.
"""
import math
import statistics

import torch

import paper_1501_06663_gb300 as lr

MI = 1 << 20
DEV = "cuda"

#: mean number of longest repeats per position (the length of the list of
#: starts over n), measured on these texts
TIES = {"english": 1.2, "dna": 1.4, "dna_iid": 1.8, "protein": 2.6, "mix": 1.7}


def listed():
    return [
        # a plasmid or a read cluster: the call's latency and its launches
        {"name": "all-dna-4k", "op": "all", "front": "sa", "kind": "dna", "n": 4099},
        # the smallest of the benchmark's strings, i.i.d. DNA: launches, look-back, few blocks
        {"name": "all-dna-1m", "op": "all", "front": "sa", "kind": "dna_iid", "n": MI},
        # a chromosome: the benchmark's planted-repeat DNA
        {"name": "all-dna-64m", "op": "all", "front": "sa", "kind": "dna", "n": 64 * MI},
        # the benchmark's headline: all longest repeats of English text
        {"name": "all-english-256m", "op": "all", "front": "sa", "kind": "english", "n": 256 * MI},
        # leftmost repeats only (no list of ties), an odd size
        {"name": "leftmost-english-100m", "op": "leftmost", "front": "sa", "kind": "english", "n": 100_000_007},
        # the paper's inputs (rank, no suffix array), a proteome: the gather front end
        {"name": "all-rank-protein-6m", "op": "all", "front": "rank", "kind": "protein", "n": 6_000_007},
        # the same on a long text: the rank windows
        {"name": "all-rank-english-80m", "op": "all", "front": "rank", "kind": "english", "n": 80_000_001},
        # many strings of uneven length in one call (an eighth of the benchmark's batched mix)
        {"name": "batch-mix-512", "op": "batch", "front": "sa", "kind": "mix", "law": "loguniform", "count": 512,
         "lo": 1024, "hi": 4 * MI},
        # one batch of the serving loop: 64 jobs of its lognormal lengths
        {"name": "batch-serving-64", "op": "batch", "front": "sa", "kind": "mix", "law": "lognormal", "count": 64,
         "lo": 1024, "hi": 16 * MI},
        # a captured plan over a few short strings, replayed
        {"name": "plan-short-24", "op": "plan", "front": "sa", "kind": "mix", "law": "loguniform", "count": 24,
         "lo": 1024, "hi": 64 * 1024},
        # host buffers in, host buffers out (the benchmark's end-to-end call), pinned memory
        {"name": "host-dna-16m", "op": "host", "front": "sa", "kind": "dna", "n": 16 * MI + 3},
        # the step before the query: suffix array, rank and lcp of a text
        {"name": "build-english-32m", "op": "build", "kind": "english", "n": 32 * MI + 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["all", "all", "all", "leftmost", "batch", "batch", "plan", "host", "build"])
    if op in ("batch", "plan"):
        law = rng.choice(["loguniform", "lognormal"])
        count = _log_int(rng, 2, 32 if op == "plan" else 400)
        hi = _log_int(rng, 4096, 256 * 1024 if op == "plan" else 4 * MI)
        return {"op": op, "front": rng.choice(["sa", "sa", "rank"]), "kind": "mix", "law": law, "count": count,
                "lo": _log_int(rng, 16, 2048), "hi": hi}
    kind = rng.choice(["english", "dna", "dna_iid", "protein"])
    if op == "build":
        return {"op": op, "kind": kind, "n": _log_int(rng, 2000, 24 * MI) | 1}
    top = {"all": 200 * MI, "leftmost": 200 * MI, "host": 16 * MI}[op]
    return {"op": op, "front": rng.choice(["sa", "sa", "rank"]), "kind": kind, "n": _log_int(rng, 2000, top)}


# ---------------------------------------------------------------- texts

def _lengths(case):
    """Lengths of a batch's strings: the quantiles of its law, whatever the seed."""
    c, lo, hi = case["count"], case["lo"], case["hi"]
    q = [(j + 0.5) / c for j in range(c)]
    if case["law"] == "loguniform":
        v = [lo * (hi / lo) ** u for u in q]
    else:
        v = [1e5 * math.exp(statistics.NormalDist().inv_cdf(u)) for u in q]
    return [max(lo, min(hi, int(x))) for x in v]


def _total(case):
    return sum(_lengths(case)) if case["op"] in ("batch", "plan") else case["n"]


def _markov_dna(n, g):
    """Order-2 Markov chains over ACGT, 256 symbols each, back to back."""
    steps = 256
    chains = (n + steps - 1) // steps
    p = torch.rand(16, 4, generator=g, device=DEV) ** 2 + 0.05
    cum = (p / p.sum(1, keepdim=True)).cumsum(1)[:, :3].contiguous()
    state = torch.randint(0, 16, (chains,), generator=g, device=DEV)
    out = torch.empty(steps, chains, dtype=torch.uint8, device=DEV)
    for t in range(steps):
        u = torch.rand(chains, 1, generator=g, device=DEV)
        nxt = (u > cum[state]).sum(1)
        out[t] = nxt
        state = (state * 4 + nxt) & 15
    return out.t().reshape(-1)[:n].contiguous()


def _slots(off, slot, g):
    """One planted stretch per `slot` positions: its slot start and the bounds of the string it lies in."""
    n = int(off[-1])
    s0 = torch.arange(0, n, slot, device=DEV)
    j = torch.searchsorted(off, s0, right=True) - 1
    return s0, off[j], torch.minimum(off[j + 1], s0 + slot), torch.rand(4, s0.numel(), generator=g, device=DEV,
                                                                        dtype=torch.float64)


def _dna(off, g):
    """DNA with about 30 % of each long string copied from elsewhere in it, 0-10 % of a copy mutated."""
    n = int(off[-1])
    text = _markov_dna(n, g)
    s0, a, e, u = _slots(off, 10500, g)
    ln = torch.minimum((300 + u[0] * 5700).long(), (e - s0).clamp(min=0))
    j = torch.searchsorted(off, s0, right=True) - 1
    ln = torch.minimum(ln, (off[j + 1] - a) // 2)
    dst = s0 + (u[1] * (e - s0 - ln + 1)).long()
    src = a + (u[2] * (off[j + 1] - a - ln + 1)).long()
    which = torch.repeat_interleave(torch.arange(s0.numel(), device=DEV), ln)
    at = torch.arange(which.numel(), device=DEV) - (ln.cumsum(0) - ln)[which]
    new = text[src[which] + at]
    hit = torch.rand(which.numel(), generator=g, device=DEV) < (0.1 * u[3]).float()[which]
    new = torch.where(hit, torch.randint(0, 4, (which.numel(),), generator=g, device=DEV, dtype=torch.uint8), new)
    text[dst[which] + at] = new
    return torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)[text.int()]


def _protein(off, g):
    """Twenty letters, about 5 % of the positions in tandem arrays (unit 3-50, 2-20 copies)."""
    n = int(off[-1])
    text = torch.tensor(list(b"ACDEFGHIKLMNPQRSTVWY"), dtype=torch.uint8, device=DEV)[
        torch.randint(0, 20, (n,), generator=g, device=DEV, dtype=torch.int32)]
    s0, _, e, u = _slots(off, 5800, g)
    unit = (3 + u[0] * 48).long()
    ln = torch.minimum(unit * (2 + u[1] * 19).long(), (e - s0).clamp(min=0))
    dst = s0 + (u[2] * (e - s0 - ln + 1)).long()
    which = torch.repeat_interleave(torch.arange(s0.numel(), device=DEV), ln)
    at = torch.arange(which.numel(), device=DEV) - (ln.cumsum(0) - ln)[which]
    text[dst[which] + at] = text[dst[which] + at % unit[which]]
    return text


def _english(n, g):
    """Words drawn by Zipf's law (s = 1.1) from 50 000, of 2-12 letters, with spaces, punctuation and newlines."""
    vocab, width = 50000, 14
    wl = torch.randint(2, 13, (vocab,), generator=g, device=DEV)
    table = torch.randint(97, 123, (vocab, width), generator=g, device=DEV, dtype=torch.uint8).reshape(-1)
    cum = (torch.arange(1, vocab + 1, device=DEV, dtype=torch.float64) ** -1.1).cumsum(0)
    words = n // 3 + 16                                # at least 3 symbols each
    w = torch.searchsorted((cum / cum[-1]).float(), torch.rand(words, generator=g, device=DEV)).clamp(max=vocab - 1)
    ul = torch.rand(words, generator=g, device=DEV)
    seps = torch.tensor([c for c in range(33, 127) if not 97 <= c <= 122], dtype=torch.uint8, device=DEV)
    mark = seps[torch.randint(0, seps.numel(), (words,), generator=g, device=DEV)]
    mark = torch.where(ul < 0.85, torch.tensor(32, dtype=torch.uint8, device=DEV), mark)
    mark = torch.where(ul > 0.99, torch.tensor(10, dtype=torch.uint8, device=DEV), mark)
    ln = wl[w] + 1 + ((ul >= 0.85) & (ul <= 0.99)).long()
    end = ln.cumsum(0)
    words = int(torch.searchsorted(end, n)) + 1
    ln, end, w, mark = ln[:words], end[:words], w[:words], mark[:words]
    which = torch.repeat_interleave(torch.arange(words, device=DEV, dtype=torch.int32), ln)[:n]
    at = torch.arange(n, device=DEV, dtype=torch.int32) - (end - ln).int()[which]
    over = at - wl.int()[w][which]                     # 0: the mark; 1: the space after punctuation
    text = table[w.int()[which] * width + at]
    text = torch.where(over == 0, mark[which], text)
    return torch.where(over == 1, torch.tensor(32, dtype=torch.uint8, device=DEV), text)


def _text(case, seed):
    """(text, offsets of its strings) on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    if case["kind"] == "mix":
        ln = torch.tensor(_lengths(case), device=DEV)
        ln = ln[torch.randperm(ln.numel(), generator=g, device=DEV)]
        off = torch.cat([ln.new_zeros(1), ln.cumsum(0)])
        isdna = torch.rand(ln.numel(), generator=g, device=DEV) < (0.7 if case["law"] == "lognormal" else 0.5)
        return torch.where(torch.repeat_interleave(isdna, ln), _dna(off, g), _protein(off, g)), off
    n = case["n"]
    off = torch.tensor([0, n], device=DEV)
    if case["kind"] == "english":
        return _english(n, g), off
    if case["kind"] == "protein":
        return _protein(off, g), off
    if case["kind"] == "dna":
        return _dna(off, g), off
    return torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)[
        torch.randint(0, 4, (n,), generator=g, device=DEV, dtype=torch.int32)], off


# ---------------------------------------------------------------- the calls

def prepare(case, seed):
    text, off = _text(case, seed)
    n, op = int(text.numel()), case["op"]
    state = {"op": op, "ctx": lr.Context(0), "n": n}
    if op == "build":
        state["text"] = text
        return state
    builder = lr.Context(0)
    try:
        if op in ("batch", "plan"):
            sa, rank, lcp = builder.build_arrays_batch(off, text)
        else:
            sa, rank, lcp = builder.build_arrays(text)
    finally:
        builder.close()
    state["sa"], state["rank"] = (sa, None) if case["front"] == "sa" else (None, rank)
    state["lcp"], state["off"] = lcp, off
    if op == "host":
        for k in ("sa", "rank", "lcp"):
            state[k] = state[k].cpu().pin_memory() if state[k] is not None else None
        where = {"pin_memory": True}
    else:
        where = {"device": DEV}
    if op != "leftmost":
        # the list of starts is shorter than its buffer; the rest of it stays zero
        state["out"] = (torch.zeros(n, dtype=torch.int32, **where), torch.zeros(n, dtype=torch.int32, **where),
                        torch.zeros(n + 1, dtype=torch.int64, **where),
                        torch.zeros(_capacity(n), dtype=torch.int32, **where))
    if op in ("batch", "plan"):
        state["desc"] = lr.batch_desc(off, lcp, sa=state["sa"], rank=state["rank"])
    if op == "plan":
        state["plan"] = _Plan(state["ctx"], state["desc"], state["out"])
    return state


def _capacity(n):
    return 4 * n + 1024


class _Plan:
    """Owns a captured plan."""

    def __init__(self, ctx, desc, out):
        self.handle = lr.lr_plan_create(ctx.handle, desc, *out)

    def __del__(self):
        lr.lr_plan_destroy(self.handle)


def run(state):
    op, ctx = state["op"], state["ctx"]
    if op == "build":
        return ctx.build_arrays(state["text"])
    sa, rank, lcp = state["sa"], state["rank"], state["lcp"]
    if op == "leftmost":
        return ctx.query_leftmost(lcp, sa=sa, rank=rank)
    out = state["out"]
    if op == "all":
        status, _ = lr.lr_query_all(ctx.handle, sa, rank, lcp, *out)
    elif op == "batch":
        status, _ = lr.lr_batch_query_all(ctx.handle, state["desc"], *out)
    elif op == "host":
        status, _ = lr.lr_query_all_host(ctx.handle, sa, rank, lcp, *out)
    else:
        lr.lr_plan_launch(state["plan"].handle)
        status, _ = lr.lr_plan_result(state["plan"].handle)
    if status != lr.LR_OK:
        raise lr.LRError(status, op)
    return out


def work(case):
    n = _total(case)
    if case["op"] == "build":
        per = 1 + 12                                   # text in; sa, rank and lcp out
    elif case["op"] == "leftmost":
        per = 8 + 8                                    # sa or rank and lcp in; lengths and starts out
    else:
        per = 8 + 16 + 4 * TIES[case["kind"]]          # and 64-bit offsets and every start out
    return {"bytes": n * per, "flops": 0}


# ---------------------------------------------------------------- plain results

def _plain_arrays(text):
    """Suffix array, rank and lcp by prefix doubling in 64-bit torch."""
    n = text.numel()
    rank, levels, h = text.long() + 1, [], 1
    while True:
        levels.append(rank)
        nxt = torch.zeros_like(rank)
        nxt[:max(0, n - h)] = rank[h:]
        key, order = torch.sort(rank * (max(n, 256) + 2) + nxt)
        step = torch.ones_like(key)
        step[1:] = (key[1:] != key[:-1]).long()
        rank = torch.empty_like(rank)
        rank[order] = step.cumsum(0)
        if int(rank.max()) == n:
            break
        h *= 2
    lcp = torch.zeros(n + 1, dtype=torch.int64, device=text.device)
    x, y, got = order[:-1].clone(), order[1:].clone(), torch.zeros(n - 1, dtype=torch.int64, device=text.device)
    for q in range(len(levels) - 1, -1, -1):
        at = torch.maximum(x, y)
        same = at < n
        lv = levels[q]
        same &= lv[x.clamp(max=n - 1)] == lv[y.clamp(max=n - 1)]
        x, y, got = x + (same << q), y + (same << q), got + (same << q)
    lcp[1:n] = got
    return order, rank - 1, lcp


def _plain_query(rank, lcp):
    """Every longest repeat: windows of the compact left-bounded repeats, taken apart position by position."""
    n, dev = rank.numel(), rank.device
    ll = torch.maximum(lcp[rank], lcp[rank + 1])
    prev = torch.cat([ll.new_zeros(1), ll[:-1]])
    cs = torch.nonzero((ll > 0) & (ll >= prev)).reshape(-1)
    ce = cs + ll[cs] - 1
    k = torch.arange(n, device=dev)
    lo, hi = torch.searchsorted(ce, k), torch.searchsorted(cs, k, right=True)
    w = (hi - lo).clamp(min=0)
    pos = torch.repeat_interleave(k, w)
    e = lo[pos] + torch.arange(pos.numel(), device=dev) - (w.cumsum(0) - w)[pos]
    length = ll[cs[e]]
    best = torch.zeros(n, dtype=torch.int64, device=dev).scatter_reduce_(0, pos, length, "amax")
    hold = length == best[pos]
    count = torch.bincount(pos[hold], minlength=n)
    offsets = torch.cat([count.new_zeros(1), count.cumsum(0)])
    starts = cs[e][hold]
    first = torch.full((n,), -1, dtype=torch.int64, device=dev)
    first[count > 0] = starts[offsets[:-1][count > 0]]
    return best, first, offsets, starts


def exact(case, seed):
    """The results of the smaller cases; all outputs are whole numbers."""
    if _total(case) > 8 * MI or case.get("count", 1) > 64:
        return None
    text, off = _text(case, seed)
    if case["op"] == "build":
        return tuple(v.int() for v in _plain_arrays(text))
    off = off.tolist()
    best, first, offsets, starts, total = [], [], [], [], 0
    for a, b in zip(off[:-1], off[1:]):
        _, rank, lcp = _plain_arrays(text[a:b])
        v = _plain_query(rank, lcp)
        best.append(v[0])
        first.append(torch.where(v[1] >= 0, v[1] + a, v[1]))
        offsets.append(v[2][:-1] + total)
        starts.append(v[3] + a)
        total += int(v[2][-1])
    offsets.append(torch.tensor([total], device=text.device))
    starts.append(starts[0].new_zeros(_capacity(text.numel()) - total))
    ln, st, of, al = torch.cat(best).int(), torch.cat(first).int(), torch.cat(offsets), torch.cat(starts).int()
    return (st, ln) if case["op"] == "leftmost" else (ln, st, of, al)
