"""SCC decomposition where the search kernels change form, against the oracle:
rows around the length that goes to the whole grid (1,024), vertex counts around
one and several CTAs, components the pivot search does not reach."""
import numpy as np
import pytest

import graphgen as gg
from tests.test_gpu_scc import check_scc

pytestmark = pytest.mark.gpu


def _P():
    import paper_2107_12720_gb300 as P
    return P


def _csr(n, u, t):
    order = np.argsort(u, kind="stable")
    off = np.zeros(n + 1, np.uint32)
    off[1:] = np.cumsum(np.bincount(u, minlength=n))
    return gg.Graph(off, np.asarray(t)[order].astype(np.uint32))


@pytest.mark.parametrize("d", [31, 32, 33, 1023, 1024, 1025, 5000])
def test_hub_rows(d):
    """A hub with d successors that all lead back to it, beside a second such
    hub that the first one reaches, and a ring that reaches both."""
    P = _P()
    ring = 7
    h1, h2 = ring, ring + 1 + d
    n = ring + 2 * (1 + d)
    u, t = [], []
    for i in range(ring):
        u += [i, i]
        t += [(i + 1) % ring, h1 + (i % d)]
    for h in (h1, h2):
        leaf = np.arange(h + 1, h + 1 + d)
        u += [h] * d + list(leaf)
        t += list(leaf) + [h] * d
    u.append(h1 + d)
    t.append(h2)
    g = _csr(n, np.array(u), np.array(t))
    with P.Trimmer(g.off, g.tgt) as tr:
        st = check_scc(tr, g, f"hubs {d}")
        assert st["components"] == 3


@pytest.mark.parametrize("n", [2, 3, 511, 512, 513, 1025, 200_003])
def test_sizes_around_the_grid(n):
    """One long cycle with chords through half the vertices, small cycles in the
    rest, random edges from the first half to the second."""
    P = _P()
    rng = np.random.default_rng(n)
    a = max(1, n // 2)
    v = np.arange(a)
    u, t = [v], [(v + 1) % a]
    u.append(rng.integers(0, a, 2 * a)); t.append(rng.integers(0, a, 2 * a))
    w = np.arange(a, n)
    if w.size:
        k = 1 + (w - a) // 5 * 0 + 4                # cycles of five (the last shorter)
        start = a + (w - a) // 5 * 5
        end = np.minimum(start + k + 1, n)
        u.append(w); t.append(np.where(w + 1 < end, w + 1, start))
        u.append(rng.integers(0, a, w.size)); t.append(w)
    g = _csr(n, np.concatenate(u), np.concatenate(t))
    with P.Trimmer(g.off, g.tgt) as tr:
        check_scc(tr, g, f"n={n}")
        check_scc(tr, g, f"n={n} again", device=True)
