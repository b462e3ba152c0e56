"""The calls by which this library's speed is measured, over the range of graphs it is used on.

Graphs follow the recipes of graphgen/configs.py (planted, R-MAT, deep cascade, batched, large
mixed) and are drawn on the GPU from the seed. Every case goes through ``Trimmer``, with the
default parameters, and reads its results back as a caller does.
"""
import math
import statistics

import torch

import paper_2107_12720_gb300 as P
from paper_2107_12720_gb300 import scheduler


def listed():
    return [
        # the smallest calls: a graph of a thousand vertices, where launches and round trips count
        dict(name="tiny_ac4", graph="planted", n=1000, op="ac4"),
        # a small graph without its transpose: sweeps over the vertices still live
        dict(name="planted_ac3", graph="planted", n=100_000, op="ac3"),
        # skewed degrees, few rounds: the ordinary call with G^T, and without it
        dict(name="rmat22_ac4", graph="rmat", n=1 << 22, op="ac4"),
        dict(name="rmat22_ac6", graph="rmat", n=1 << 22, op="ac6"),
        # vertex sampling (the scalability experiment): a new dead mask before the run
        dict(name="sampled_ac4", graph="rmat", n=3_000_017, op="sampled", share=0.5),
        # one graph used once: context, transpose, run, result, all in the call
        dict(name="oneshot_ac4", graph="rmat", n=1 << 22, op="oneshot"),
        # the decomposition that trimming feeds
        dict(name="rmat20_scc", graph="rmat", n=1 << 20, op="scc"),
        # deep peeling: thousands of short rounds, with and without G^T
        dict(name="deep24_ac4", graph="deep", n=1 << 24, chain=2867, op="ac4"),
        dict(name="deep_ac6", graph="deep", n=1_000_003, chain=1500, op="ac6"),
        # size-1 components of a deep graph (both degrees checked), a ragged size
        dict(name="deep_inout", graph="deep", n=5_000_011, chain=2001, op="inout"),
        # thousands of independent graphs packed into one call
        dict(name="batch4096_ac4", graph="batch", graphs=4096, op="batch"),
        # the largest graph: R-MAT scale 26 and a block of 10,000-deep chains, learned schedule
        dict(name="mixed_learned", graph="mixed", n=1 << 26, block=1 << 25, chain=10_000,
             op="learned"),
    ]


def _spread(rng, lo, hi):
    """A size between lo and hi, uniform in its logarithm (any remainder)."""
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["planted", "planted", "rmat", "rmat", "rmat", "deep", "deep", "batch",
                       "mixed"])
    if kind == "planted":
        op = rng.choice(["ac4", "ac3"])
        return dict(graph=kind, n=_spread(rng, 1000, 4_000_000 if op == "ac4" else 400_000), op=op)
    if kind == "rmat":
        op = rng.choice(["ac4", "ac6", "sampled", "oneshot", "scc"])
        c = dict(graph=kind, n=_spread(rng, 1 << 14, 1 << (20 if op == "scc" else 22)), op=op)
        if op == "sampled":
            c["share"] = round(rng.uniform(0.1, 0.9), 2)
        return c
    if kind == "deep":
        op = rng.choice(["ac4", "ac6", "inout"])
        top = {"ac4": 1 << 24, "ac6": 1 << 20, "inout": 1 << 23}[op]
        return dict(graph=kind, n=_spread(rng, 1 << 16, top), chain=_spread(rng, 200, 2867), op=op)
    if kind == "batch":
        return dict(graph=kind, graphs=_spread(rng, 64, 4096), op="batch")
    n = _spread(rng, 1 << 17, 1 << 25)
    return dict(graph=kind, n=n, block=_spread(rng, n // 4, n // 2), chain=_spread(rng, 300, 5000),
                op="learned")


# ------------------------------------------------------------------ graphs


def _blocks(case):
    """The planted blocks of a case, one row per independent graph: sizes of the core C, the
    reaching set R and the trimmable set T, sinks of T, degree ranges of C, R and T, chains."""
    if case["graph"] == "planted":
        n = case["n"]
        c, r = n * 3 // 10, n * 3 // 10
        t = n - c - r
        return [(c, r, t, max(1, t // 20), 4, 4, 1, 4, 1, 4, 0)]
    if case["graph"] in ("deep", "mixed"):
        n = case["n"] if case["graph"] == "deep" else case["block"]
        c, r = n // 10, n // 5
        t = n - c - r
        return [(c, r, t, 0, 8, 8, 1, 15, 0, 14, max(1, t // case["chain"]))]
    if case["graph"] == "batch":  # log-normal sizes (median 2,000, sigma 1.5), degrees 2..12
        rows, z = [], statistics.NormalDist()
        for i in range(case["graphs"]):
            n = round(2000 * math.exp(1.5 * z.inv_cdf((i + 0.5) / case["graphs"])))
            n = max(64, min(2_000_000, n))
            d = 2 + (i * 7919) % 11
            t = int(0.9 * ((i * 0.6180339887498949) % 1.0) * n)
            c = max(1, (n - t) // 2)
            rows.append((c, n - t - c, t, -(-t // 20), 1, 2 * d - 1, 1, 2 * d - 1, 1, 2 * d - 1, 0))
        return rows
    return []


def _uniform(gen, k):
    """Uniform integers below each entry of k."""
    return (torch.rand(k.shape, generator=gen, device="cuda", dtype=torch.float64) * k).long()


def _planted_edges(gen, rows):
    """Edges of the disjoint union of planted blocks (see include/trim.h for the recipe)."""
    b = torch.tensor(rows, device="cuda", dtype=torch.int64)
    size = b[:, 0] + b[:, 1] + b[:, 2]
    start = torch.cumsum(size, 0) - size
    g = torch.repeat_interleave(torch.arange(len(rows), device="cuda"), size)
    v = torch.arange(g.numel(), device="cuda") - start[g]
    nc, ncr, chains = b[g, 0], b[g, 0] + b[g, 1], b[g, 10]
    in_c, in_t = v < nc, v >= ncr
    lo = torch.where(in_c, b[g, 4], torch.where(in_t, b[g, 8], b[g, 6]))
    hi = torch.where(in_c, b[g, 5], torch.where(in_t, b[g, 9], b[g, 7]))
    deg = lo + _uniform(gen, hi - lo + 1)
    rank = v - ncr
    chained = in_t & (chains > 0)
    deg = torch.where(chained, deg + 1, deg)
    deg[in_t & (rank < torch.where(chains > 0, chains, b[g, 3]))] = 0
    u = torch.repeat_interleave(torch.arange(g.numel(), device="cuda"), deg)
    first = torch.arange(u.numel(), device="cuda") == (torch.cumsum(deg, 0) - deg)[u]
    # targets: C and the first of R in C, the rest of R in C and R, T below its own rank (a chain
    # link: its chain predecessor first, the others at lower positions)
    pos = torch.where(chains > 0, rank - rank % chains.clamp(min=1), rank)
    top = torch.where(in_c, nc, torch.where(in_t, pos, ncr))
    span = torch.where(first & ~in_t[u], nc[u], top[u])
    t = _uniform(gen, span) + torch.where(in_t, ncr, 0)[u]
    t = torch.where(first & chained[u], v[u] - chains[u], t) + start[g][u]
    return u, t


def _rmat_edges(gen, n):
    """R-MAT edges (.57, .19, .19, .05), 16 draws per vertex, folded onto n permuted ids; a tenth
    of the vertices lose their out-edges."""
    src = torch.zeros(16 * n, dtype=torch.int32, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(max(1, (n - 1).bit_length())):
        x = torch.rand(16 * n, generator=gen, device="cuda")
        down = x >= 0.76
        right = ((x >= 0.57) & ~down) | (x >= 0.95)
        src.mul_(2).add_(down)
        dst.mul_(2).add_(right)
    perm = torch.randperm(n, generator=gen, device="cuda", dtype=torch.int64)
    src, dst = perm[src.remainder_(n)], perm[dst.remainder_(n)]
    sink = torch.zeros(n, dtype=torch.bool, device="cuda")
    sink[torch.randperm(n, generator=gen, device="cuda")[:n // 10]] = True
    keep = (src != dst) & ~sink[src]
    return src[keep], dst[keep]


def _csr(key, n):
    """Rows and targets, as int32, of sorted keys row * n + target."""
    row = torch.div(key, n, rounding_mode="floor")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=off[1:])
    return off.to(torch.int32), (key - row * n).to(torch.int32)


def _graph(case, seed, transposed):
    """(off, tgt) and, if asked for, (off_in, tgt_in): sorted rows, no edge twice."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 2654435761 % (1 << 62) + 17)
    parts, n = [], 0
    if case["graph"] in ("rmat", "mixed"):
        parts.append(_rmat_edges(gen, case["n"]))
        n = case["n"]
    rows = _blocks(case)
    if rows:
        u, t = _planted_edges(gen, rows)
        nb = sum(r[0] + r[1] + r[2] for r in rows)
        if case["graph"] == "deep":  # where C begins: a level is a chain position whatever the seed
            turn = int(torch.randint(nb, (1,), generator=gen, device="cuda"))
            u, t = (u + turn) % nb, (t + turn) % nb
        parts.append((u + n, t + n))
        n += nb
    key = torch.cat([u * n + t for u, t in parts])
    del parts
    key = torch.sort(key).values
    key = torch.unique_consecutive(key)
    out = _csr(key, n)
    if not transposed:
        return n, out, (None, None)
    row = torch.div(key, n, rounding_mode="floor")
    key = torch.sort((key - row * n) * n + row).values
    del row
    return n, out, _csr(key, n)


# ------------------------------------------------------------------ the calls


def _sampled_away(case, seed, n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 40503 + 99)
    return torch.rand(n, generator=gen, device="cuda") >= case["share"]


def prepare(case, seed):
    op = case["op"]
    n, (off, tgt), (ioff, itgt) = _graph(case, seed, op not in ("ac6", "ac3", "oneshot"))
    s = dict(op=op)
    if op == "oneshot":
        s["csr"] = (off, tgt)
        return s
    s["t"] = P.Trimmer(off, tgt, ioff, itgt)
    if op == "learned":
        s["t"].set_model(scheduler.load_blob())
    if op == "sampled":
        s["mask"] = _sampled_away(case, seed, n)
    if op == "batch":
        ends = torch.tensor([0] + [r[0] + r[1] + r[2] for r in _blocks(case)]).cumsum(0)
        s["graph_off"] = ends.numpy().astype("uint32")
    return s


def _levels(t, st):
    return dict(level=t.level().view(torch.int32), rounds=st["rounds"], dead=st["n_dead"])


def run(state):
    op = state["op"]
    if op == "oneshot":
        with P.Trimmer(*state["csr"]) as t:
            return _levels(t, t.run("ac4"))
    t = state["t"]
    if op == "scc":
        comp, st = t.run_scc(device=True)
        return dict(comp=comp, components=st["components"])
    if op == "inout":
        return _levels(t, t.run_inout())
    if op == "batch":
        return _levels(t, t.batch_run(state["graph_off"], "ac4"))
    if op == "sampled":
        t.set_dead_mask(state["mask"])
        out = _levels(t, t.run("ac4"))
        return dict(out, status=t.status())
    return _levels(t, t.run(op))


def work(case):
    """Bytes of one pass: the offsets, the edges the path has to see, the results; all 32-bit."""
    rows = _blocks(case)
    n = sum(r[0] + r[1] + r[2] for r in rows)
    removed = sum(r[2] for r in rows)
    edges = sum((r[2] - (r[10] or r[3])) * ((r[8] + r[9]) / 2 + (1 if r[10] else 0)) for r in rows)
    m = edges + sum(r[0] * (r[4] + r[5]) / 2 + r[1] * (r[6] + r[7]) / 2 for r in rows)
    if case["graph"] in ("rmat", "mixed"):
        # shares that the recipe gives at scale 22: vertices removed, their in-edges, all edges
        n, removed = n + case["n"], removed + 0.58 * case["n"]
        edges, m = edges + 1.57 * case["n"], m + 13.9 * case["n"]
    op = case["op"]
    if op in ("ac4", "learned", "batch"):  # G^T rows of the removed vertices
        b = 4 * n + 8 * removed + 4 * edges + 4 * n
    elif op in ("ac6", "ac3"):  # rows of the removed vertices, one live successor of the others
        own = 0 if case["graph"] == "rmat" else edges
        b = 4 * n + 4 * own + 4 * (n - removed) + 4 * n
    elif op == "inout":  # both offsets, both rows of the removed vertices
        b = 8 * n + 8 * edges + 4 * n
    elif op == "sampled":  # the mask, the rows of the sampled vertices, levels and status
        b = n + 4 * n + 4 * case["share"] * m + 4 * case["share"] ** 2 * edges + 5 * n
    elif op == "scc":  # both CSRs, the labels
        b = 8 * n + 8 * m + 4 * n
    else:  # oneshot: the CSR, the levels
        b = 4 * n + 4 * m + 4 * n
    return {"bytes": float(b), "flops": 0.0}


# ------------------------------------------------------------------ what the results are


def _peel(n, off, ioff, itgt, gone=None):
    """Levels by definition: a vertex goes one step after the last of its successors."""
    left = (off[1:] - off[:-1]).clone() if gone is None else gone
    level = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    front = torch.nonzero(left == 0).flatten()
    step = 0
    while front.numel():
        level[front] = step
        lo = ioff[front].long()
        k = ioff[front + 1].long() - lo
        end = torch.cumsum(k, 0)
        at = torch.arange(int(end[-1]), device="cuda") + torch.repeat_interleave(lo - end + k, k)
        p = itgt[at].long()
        left.scatter_add_(0, p, torch.full_like(p, -1, dtype=left.dtype))
        front = torch.unique(p[left[p] == 0])
        step += 1
    return level


def _told(level, masked=None):
    dead = level != -1
    if masked is not None:
        dead &= ~masked
    top = int(level[dead].max()) + 1 if bool(dead.any()) else 0
    return dict(level=level, rounds=top, dead=int(dead.sum()))


def exact(case, seed):
    op = case["op"]
    if op == "scc":
        return None
    n, (off, tgt), (ioff, itgt) = _graph(case, seed, True)
    if op == "inout":  # whichever of the two peelings reaches a vertex first
        a, b = _peel(n, off, ioff, itgt), _peel(n, ioff, off, tgt)
        return _told(torch.where(a == -1, b, torch.where(b == -1, a, torch.minimum(a, b))))
    if op != "sampled":
        return _told(_peel(n, off, ioff, itgt))
    away = _sampled_away(case, seed, n)
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), (off[1:] - off[:-1]).long())
    keep = ~away[src] & ~away[tgt.long()]
    u, t = src[keep], tgt.long()[keep]
    left = torch.bincount(u, minlength=n).to(torch.int32)
    left[away] = -1  # never reaches zero
    key = torch.sort(t * n + u).values
    sub_off, sub_tgt = _csr(key, n)
    out = _told(_peel(n, off, sub_off, sub_tgt, left))
    out["level"] = torch.where(away, torch.full_like(out["level"], -2), out["level"])
    return dict(out, status=(out["level"] == -1).to(torch.uint8))
