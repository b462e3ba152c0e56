"""In+out trimming of shallow graphs whose first round removes far more vertices than there
are warps, with few edges in all: that round is an ordinary one (a local round would give
every warp tens of rows, one after the other), later ones may be local."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sinks", [100, 60_000])
def test_wide_rounds_are_ordinary(sinks):
    """`sinks` vertices without successors, two predecessors each out of a second layer; a
    chain of 20 above it, and a cycle that stays."""
    import paper_2107_12720_gb300 as P
    rng = np.random.default_rng(sinks)
    rows = [[] for _ in range(sinks)]
    second = sinks // 2
    for _ in range(second):
        rows.append(list(rng.integers(0, sinks, 4)))
    for i in range(20):
        rows.append([len(rows) - 1])
    c = len(rows)
    rows += [[c + 1, c - 1], [c + 2], [c]]
    g = gg.edges_from_lists(len(rows), rows)
    csr_in = oracle.transpose(g.off, g.tgt)
    level, status, alpha = oracle.peel_inout(g.off, g.tgt, csr_in)
    with P.Trimmer(g.off, g.tgt, *csr_in) as t:
        s = t.run_inout()
        assert np.array_equal(t.level(device=False), level)
        assert np.array_equal(t.status(device=False), status)
        assert s["rounds"] == alpha and s["n_dead"] == int((status == 0).sum())
        assert (s["local_rounds"] < alpha) == (sinks > 10_000)
        assert s["local_rounds"] > 0
