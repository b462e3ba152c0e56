"""AC-6 and AC-3 on rows read in place from host memory, where AC-6's records leave the next
successor unread: rows of one, two and many successors, supports that go early and late,
with local rounds and without, against the oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _graph(n, most, stay, seed):
    """Rows of 0 to `most` successors below the vertex; a share `stay` also reaches a cycle,
    as the last successor."""
    rng = np.random.default_rng(seed)
    rows = [[1], [0]]
    for v in range(2, n):
        r = list(rng.integers(2, v, rng.integers(0, most + 1))) if v > 2 else []
        if rng.random() < stay:
            r.append(int(rng.integers(0, 2)))
        rows.append(r)
    return gg.edges_from_lists(n, rows)


@pytest.mark.parametrize("n,most,stay", [(500, 1, 0.0), (2000, 2, 0.1), (5000, 9, 0.3),
                                         (3000, 70, 0.02), (30_000, 4, 0.05)])
def test_against_the_oracle(n, most, stay):
    import torch
    import paper_2107_12720_gb300 as P
    g = _graph(n, most, stay, n)
    level, status, alpha = oracle.peel(g.off, g.tgt)[:3]
    pin = lambda a: torch.from_numpy(a.astype(np.int32)).pin_memory()
    with P.Trimmer(pin(g.off), pin(g.tgt), host_mapped=True) as t:
        for local in (None, 0):
            if local is not None:
                t.set_params(local_round_edges=local)
            for v in ("ac6", "ac3", "ac6"):
                s = t.run(v)
                assert np.array_equal(t.level(device=False), level), (v, local)
                assert np.array_equal(t.status(device=False), status), (v, local)
                assert s["rounds"] == alpha and s["n_dead"] == int((status == 0).sum())
