"""The asynchronous AC-4 tail where its handovers change form, against the oracle.

A worker warp keeps one row of at most 32 in-edges and hands the others on: rows
of a batch go to idle workers or the CTA's ring, longer ones in pieces of 32, rows
over 1,024 in-edges to the global pieces (256 each). A level with about more
vertices than there are workers keeps rounds, and the tail starts later.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.test_gpu_parity import check

pytestmark = pytest.mark.gpu


def _P():
    import paper_2107_12720_gb300 as P
    return P


def _rows_along_a_chain(sizes, start=132, length=240):
    """A chain c_{length-1} -> ... -> c_0 whose vertices from `start` on have
    sizes[i % len] in-edges besides the chain's, from leaves of out-degree 1."""
    k = np.array([sizes[i % len(sizes)] if i >= start else 1 for i in range(length)], np.int64)
    leaf = np.repeat(np.arange(length, dtype=np.uint32), k)
    deg = np.ones(length + leaf.size, np.int64)
    deg[0] = 0
    off = np.zeros(deg.size + 1, np.uint32)
    off[1:] = np.cumsum(deg)
    return off, np.concatenate([np.arange(length - 1, dtype=np.uint32), leaf])


@pytest.mark.parametrize("block", [512, 128])
@pytest.mark.parametrize("sizes", [(0, 1), (30, 31, 32, 33), (62, 63, 64, 65),
                                   (1022, 1023, 1024, 1025), (255, 256, 257, 5000)])
def test_rows_around_the_piece_sizes(sizes, block):
    P = _P()
    off, tgt = _rows_along_a_chain(sizes)
    lvl, st, alpha = oracle.peel(off, tgt)
    assert alpha >= 240
    with P.Trimmer(off, tgt, flags=P.TRIM_FLAG_STATS) as t:
        t.set_params(block_threads=block)
        for rep in range(3):
            s = t.run("ac4")
            check(t, lvl, st, alpha, f"{sizes}-{block}-{rep}", s)
            assert s["async_round"] == 128 and s["in_edges_pushed"] == off.size - 2


@pytest.mark.parametrize("chains,length", [(1, 700), (33, 500), (600, 400), (4000, 300)])
def test_coupled_chains(chains, length):
    """Chains whose links also point to near lower positions of other chains: the
    last successor to go is seldom the chain's own, so rows change hands all the time."""
    P = _P()
    rng = np.random.default_rng(chains)
    n = chains * length
    v = np.arange(chains, n)
    u, t = [v], [v - chains]
    for _ in range(5):
        pos = v // chains
        back = 1 + rng.integers(0, np.minimum(pos, 12))
        u.append(v)
        t.append((pos - back) * chains + rng.integers(0, chains, v.size))
    u, t = np.concatenate(u), np.concatenate(t)
    order = np.argsort(u, kind="stable")
    off = np.zeros(n + 1, np.uint32)
    off[1:] = np.cumsum(np.bincount(u, minlength=n))
    tgt = t[order].astype(np.uint32)
    lvl, st, alpha = oracle.peel(off, tgt)
    assert alpha == length
    with P.Trimmer(off, tgt) as tr:
        for rep in range(3):
            check(tr, lvl, st, alpha, f"coupled-{chains}-{rep}", tr.run("ac4"))


def test_tail_starts_once_the_levels_are_small():
    """20,000 chains of 150 levels beside 300 of 420: rounds while both run, the
    tail for the rest."""
    P = _P()
    g = gg.union([gg.planted(1, 100, 100, 20000 * 150, t_k=(0, 2), n_chains=20000),
                  gg.planted(2, 100, 100, 300 * 420, t_k=(0, 2), n_chains=300, salt=1 << 40)])
    lvl, st, alpha = oracle.peel(g.off, g.tgt)
    with P.Trimmer(g.off, g.tgt) as t:
        s = t.run("ac4")
        check(t, lvl, st, alpha, "late tail", s)
        assert s["async_round"] > 150
        assert s["async_removed"] == int(((lvl >= s["async_round"]) & (st == 0)).sum())
