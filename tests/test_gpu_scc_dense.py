"""SCC decomposition of many rows over 1,024 edges, the length from which a frontier's rows
are cut into pieces and spread over the grid, against the oracle: dense parts joined by
single edges, so that the label propagation and the backward searches (which start from
every open vertex) meet all rows at once."""
import numpy as np
import pytest

import graphgen as gg
from tests.test_gpu_scc import check_scc

pytestmark = pytest.mark.gpu


def dense_parts(parts, size, degrees, seed):
    """`parts` strongly connected parts of `size` vertices, vertex i of a part with
    degrees[i % len(degrees)] successors in it; each part has one edge to the next."""
    rng = np.random.default_rng(seed)
    n = parts * size
    deg = np.resize(np.asarray(degrees), n).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(deg)])
    first = np.arange(n) // size * size
    tgt = np.repeat(first, deg) + rng.integers(0, size, off[-1])
    tgt[off[:-1]] = first + (np.arange(n) - first + 1) % size  # a ring through the part
    joint = np.arange(parts - 1) * size
    tgt[off[joint] + 1] = joint + size
    return gg.Graph(off.astype(np.uint32), tgt.astype(np.uint32))


@pytest.mark.parametrize("parts,size,degrees", [
    (2, 700, [1025]), (3, 1100, [1024, 1025]), (5, 1300, [1280, 1281, 20]),
    (4, 1500, [2000, 1536, 1537, 1024, 3])])
def test_rows_cut_into_pieces(parts, size, degrees):
    import paper_2107_12720_gb300 as P
    g = dense_parts(parts, size, degrees, parts)
    with P.Trimmer(g.off, g.tgt) as t:
        st = check_scc(t, g, f"{parts} x {size}")
        assert st["components"] == parts
        check_scc(t, g, "again", device=True)


def test_thousands_of_rows_share_the_grid():
    """12,000 rows of 1,100 edges. A CTA waits for the others at the end of a phase for at
    most spin_limit_ns; with the rows spread over the grid a phase takes some 100 us, with
    each row on the first warps alone some 50 ms."""
    import paper_2107_12720_gb300 as P
    g = dense_parts(8, 1500, [1100], 1)
    with P.Trimmer(g.off, g.tgt) as t:
        t.in_csr()
        t.set_params(spin_limit_ns=10_000_000)
        st = check_scc(t, g, "12,000 long rows")
        assert st["components"] == 8 and st["fwbw_steps"] > 1


def test_a_long_phase_is_not_a_timeout():
    """A vertex with four million removed successors and one open one, the other half of its
    size-2 component: one warp reads that row for some 100 ms, far longer than the limit of a
    wait without progress (the in+out trimming before it takes about 5 ms)."""
    import paper_2107_12720_gb300 as P
    k = 1 << 22
    off = np.zeros(k + 3, np.uint32)
    off[k + 1] = k + 1
    off[k + 2] = k + 2
    tgt = np.concatenate([np.arange(k), [k + 1, k]]).astype(np.uint32)
    with P.Trimmer(off, tgt) as t:
        t.in_csr()
        assert t.run_inout()["device_ms"] < 15
        t.set_params(spin_limit_ns=30_000_000)
        comp, st = t.run_scc()
        assert st["ms"] > 60  # the phase is longer than the limit
        want = np.arange(k + 2, dtype=np.uint32)
        want[k + 1] = k
        assert np.array_equal(comp, want)
        assert st["components"] == k + 1 and st["trimmed_size2"] == 1
