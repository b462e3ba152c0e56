"""In+out trimming on the GPU at the edges of its local rounds: rows at the
length that still fits a CTA's queue and one past it, more pushes in one round
than the queues take, vertices that both directions remove in the same round,
and the same graphs with local rounds off, element by element against the
oracle's peel_inout."""

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def layered(widths, fan, seed):
    """Layers of the given widths; every vertex has `fan` edges into the layer below (itself a
    sink layer at the bottom), some layers also a few edges to any lower layer."""
    rng = np.random.default_rng(seed)
    start = np.concatenate([[0], np.cumsum(widths)])
    rows = [[] for _ in range(int(start[-1]))]
    for k in range(1, len(widths)):
        for v in range(start[k], start[k + 1]):
            f = fan if isinstance(fan, int) else fan[k]
            rows[v] = list(rng.integers(start[k - 1], start[k], f))
            if k % 3 == 0:
                rows[v] += list(rng.integers(0, start[k], 2))
    return gg.edges_from_lists(len(rows), rows)


def star_layers(width, layers):
    """Alternating hubs and leaves: each hub has `width` in- and out-edges."""
    rows, hub = [], 0
    rows.append([])
    for _ in range(layers):
        leaves = range(len(rows), len(rows) + width)
        rows += [[hub] for _ in leaves]
        hub = len(rows)
        rows.append(list(leaves))
    return gg.edges_from_lists(len(rows), rows)


def with_core(g, seed):
    """g with a cycle of ten vertices in its middle: some vertices stay."""
    off, tgt = g.off.astype(np.int64), g.tgt.astype(np.int64)
    n = off.size - 1
    rows = [list(tgt[off[v]:off[v + 1]]) for v in range(n)]
    rng = np.random.default_rng(seed)
    mid = n // 2
    for i in range(10):
        rows.append([n + (i + 1) % 10])
        rows[n + i].append(int(rng.integers(0, mid)))
        rows[int(rng.integers(mid, n))].append(n + i)
    return gg.edges_from_lists(len(rows), rows)


CASES = {
    "row 64": lambda: star_layers(64, 40),
    "row 65": lambda: star_layers(65, 40),
    "row 256": lambda: star_layers(256, 8),
    "row 257": lambda: star_layers(257, 8),
    "chain": lambda: layered([1] * 301, 1, 1),
    "even layers meet in one round": lambda: layered([5] * 100, 3, 2),
    "odd layers": lambda: layered([5] * 101, 3, 3),
    "queues overflow": lambda: layered([2000, 15000, 30000, 15000, 2000] * 2, 4, 4),
    "narrow then wide": lambda: layered([1] * 20 + [3000] * 20 + [1] * 20, 5, 5),
}


@pytest.mark.parametrize("core", [False, True])
@pytest.mark.parametrize("name", list(CASES))
def test_against_the_oracle(name, core):
    import paper_2107_12720_gb300 as P
    g = CASES[name]()
    if core:
        g = with_core(g, 7)
    csr_in = oracle.transpose(g.off, g.tgt)
    level, status, alpha = oracle.peel_inout(g.off, g.tgt, csr_in)
    dead = status == 0
    with P.Trimmer(g.off, g.tgt, *csr_in, flags=P.TRIM_FLAG_STATS) as t:
        for local in (None, 0):
            if local is not None:
                t.set_params(local_round_edges=local)
            s = t.run_inout()
            assert np.array_equal(t.level(device=False), level), (name, local)
            assert np.array_equal(t.status(device=False), status), (name, local)
            assert s["rounds"] == alpha and s["n_dead"] == int(dead.sum())
            assert s["in_edges_pushed"] == int(np.diff(csr_in[0].astype(np.int64))[dead].sum())
            assert s["edges_inspected"] == int(np.diff(g.off.astype(np.int64))[dead].sum())
            if local == 0:
                assert s["local_rounds"] == 0
            elif name == "chain":
                assert s["local_rounds"] > 0
