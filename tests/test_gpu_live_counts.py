"""Work counters of AC-3 alone with a live list per CTA: each round's list entries and edges are
added to the run's totals when the round ends."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_live_lists import KEEP, cascade

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 9727, 100_003])
@pytest.mark.parametrize("threads", [128, 512])
def test_every_round_counts_the_vertices_still_live(n, threads):
    import paper_2107_12720_gb300 as P
    g = cascade(n, n, KEEP["every third block"])
    level, status, alpha = oracle.peel(g.off, g.tgt)[:3]
    left = np.where(status == 1, np.uint32(0xFFFFFFFF), level)
    # (no round runs if step 0 removes nothing)
    want = n + sum(int((left >= r).sum()) for r in range(2, alpha + 1)) if alpha else 0
    with P.Trimmer(g.off, g.tgt, flags=P.TRIM_FLAG_STATS) as t:
        t.set_params(block_threads=threads, ctas_per_sm=1)
        for _ in range(2):
            s = t.run("ac3")
            assert np.array_equal(t.level(device=False), level)
            assert s["live_swept"] == want
            assert s["edges_inspected"] >= want - n
