"""AC-3 on the GPU with a live list per CTA, against the oracle: vertex counts
around a block of 32, a CTA's warps and a turn of the whole grid (where parts of the
lists differ by a block), vertices that survive in some blocks only, a dead mask,
the same runs with shared lists, with other CTA sizes and on repeated calls."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def cascade(n, seed, keep):
    """Vertices over a cycle of five: each has up to seven successors below it; those in the
    blocks of 32 that `keep` picks also reach the cycle and stay."""
    rng = np.random.default_rng(seed)
    rows = [[(i + 1) % 5] for i in range(5)]
    for v in range(5, n):
        succ = list(rng.integers(5, v, int(rng.integers(0, 8)))) if v > 5 else []
        if keep(v // 32):
            succ.append(int(rng.integers(0, 5)))
        rows.append(succ)
    return gg.edges_from_lists(n, rows)


KEEP = {"none": lambda b: False, "every third block": lambda b: b % 3 == 0,
        "the first blocks": lambda b: b < 40}
SIZES = [6, 31, 32, 33, 511, 513, 4864, 4865, 9727]


@pytest.mark.parametrize("keep", list(KEEP))
@pytest.mark.parametrize("n", SIZES)
def test_against_the_oracle(n, keep):
    import paper_2107_12720_gb300 as P
    g = cascade(n, n, KEEP[keep])
    level, status, alpha = oracle.peel(g.off, g.tgt)[:3]
    with P.Trimmer(g.off, g.tgt) as t:
        for params in ({}, {"block_threads": 160}, {"ctas_per_sm": 1, "block_threads": 512},
                       {"local_round_edges": 0}):
            t.set_params(**params)
            for _ in range(2):
                s = t.run("ac3")
                assert np.array_equal(t.level(device=False), level), (n, keep, params)
                assert np.array_equal(t.status(device=False), status), (n, keep, params)
                assert s["rounds"] == alpha and s["n_dead"] == int((status == 0).sum())


def test_more_vertices_than_a_turn_with_a_mask():
    import paper_2107_12720_gb300 as P
    g = cascade(160_001, 3, lambda b: b % 5 == 2)
    mask = np.random.default_rng(4).random(160_001) < 0.3
    level, status = oracle.peel_masked(g.off, g.tgt, mask)[:2]
    with P.Trimmer(g.off, g.tgt) as t:
        t.set_dead_mask(mask.astype(np.uint8))
        t.run("ac3")
        assert np.array_equal(t.level(device=False), level)
        assert np.array_equal(t.status(device=False), status)
