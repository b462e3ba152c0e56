"""A call that finds too little device memory keeps none of it: however often it is repeated,
the smallest cap that lets it succeed stays the same."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _graph():
    """Few vertices, many edges: the last of in+out trimming's arrays is its largest."""
    n, d = 2000, 400
    off = (np.arange(n + 1) * d).astype(np.uint32)
    tgt = np.random.default_rng(1).integers(0, n, n * d).astype(np.uint32)
    return gg.Graph(off, tgt)


def test_inout_out_of_memory_again_and_again():
    import paper_2107_12720_gb300 as P
    g = _graph()
    csr_in = oracle.transpose(g.off, g.tgt)

    def succeeds(limit, before=0):
        with P.Trimmer(g.off, g.tgt, *csr_in) as t:
            try:
                for cap in [limit - 256] * before + [limit]:
                    P.trim_set_alloc_limit(cap)
                    try:
                        t.run_inout()
                        ok = True
                    except P.TrimError as e:
                        assert e.code == 4
                        ok = False
                return ok
            finally:
                P.trim_set_alloc_limit(0)

    lo, hi = 0, 1 << 30  # (the caps of a fresh context that fail, and succeed)
    assert succeeds(hi)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if succeeds(mid) else (mid, hi)
    assert not succeeds(hi - 256)
    assert succeeds(hi, before=20)
