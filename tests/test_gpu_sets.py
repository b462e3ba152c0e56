"""AC-6 on the GPU where its sets change form, against the oracle: sets around the
32 members of a re-scan, built at the start or joined later (four lists by a
hash), members that move from support to support, more removals in a round than the
CTAs' queues take, supports that contend for a slot of the counting table, vertex
counts around the block sizes, and the same graphs with local rounds off and with
small CTAs."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def bulk_star(k):
    """k leaves on a hub that is removed in round 1, behind each leaf one more vertex."""
    rows = [[], [0]] + [[1]] * k + [[2 + i] for i in range(k)]
    return gg.edges_from_lists(len(rows), rows)


def joined_star(k, length):
    """k vertices whose successors are the vertices of one chain in order: all of them
    move along the chain, one list of k members at a time."""
    rows = [[]] + [[i] for i in range(length)]
    rows += [list(range(length + 1)) for _ in range(k)]
    return gg.edges_from_lists(len(rows), rows)


def cascade(n, chains, core, seed):
    """Layers of `chains` vertices over `core` vertices of a cycle; each has its predecessor in
    the layer below and random vertices of lower layers as successors, sorted."""
    rng = np.random.default_rng(seed)
    rows = [[(i + 1) % core] for i in range(core)]
    for i in range(n - core):
        if i < chains:
            rows.append([])
            continue
        low = core + i - i % chains
        k = int(rng.integers(0, 8))
        rows.append(sorted([core + i - chains] + list(rng.integers(core, low, k))))
    for v in rng.integers(core, n, (n - core) // 50):  # these and all above them stay
        rows[int(v)].insert(0, 0)
    return gg.edges_from_lists(n, rows)


def wide_cascade(seed):
    """Layers of very different widths: the queues of some rounds overflow."""
    rng = np.random.default_rng(seed)
    rows, prev = [], []
    for width in [400, 400, 6000, 20, 20, 6000, 1, 1, 900] * 3:
        ids = range(len(rows), len(rows) + width)
        rows += [list(rng.choice(prev, 3)) if len(prev) else [] for _ in ids]
        prev = np.arange(ids.start, ids.stop)
    return gg.edges_from_lists(len(rows), rows)


CASES = {f"bulk {k}": (lambda k=k: bulk_star(k)) for k in (1, 31, 32, 33, 64, 65, 5000)}
CASES.update({f"joined {k}": (lambda k=k: joined_star(k, 40)) for k in (1, 3, 31, 32, 33, 130, 700)})
CASES.update({f"cascade {n}": (lambda n=n: cascade(n, 37, 5, n)) for n in (127, 128, 130, 511, 6001)})
CASES["wide cascade"] = lambda: wide_cascade(1)
CASES["narrow cascade"] = lambda: cascade(3000, 3, 0, 2)


@pytest.mark.parametrize("name", list(CASES))
def test_against_the_oracle(name):
    import paper_2107_12720_gb300 as P
    g = CASES[name]()
    level, status, alpha = oracle.peel(g.off, g.tgt)[:3]
    with P.Trimmer(g.off, g.tgt) as t:
        for params in ({}, {"local_round_edges": 0},
                       {"local_round_edges": 1 << 18, "block_threads": 160}):
            t.set_params(**params)
            for _ in range(2):
                s = t.run("ac6")
                assert np.array_equal(t.level(device=False), level), (name, params)
                assert np.array_equal(t.status(device=False), status), (name, params)
                assert s["rounds"] == alpha and s["n_dead"] == int((status == 0).sum())
