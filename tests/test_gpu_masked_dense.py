"""Vertex-sampled AC-4 runs where the masked initial pass changes form, against the oracle's
peel_masked: rows around the lengths that a warp (512) or the whole CTA (2,048) takes, more
long rows than a CTA's list holds, vertex counts around those from which targets pass by the
L1 (2^21); and a small graph of long rows keeps all SMs at work."""
import numpy as np
import pytest

import graphgen as gg
from tests.test_gpu_masked import check_masked

pytestmark = pytest.mark.gpu


def _graph(n, degrees, seed):
    rng = np.random.default_rng(seed)
    deg = np.resize(np.asarray(degrees), n).astype(np.int64)
    deg[rng.random(n) < 0.1] = 0
    off = np.concatenate([[0], np.cumsum(deg)])
    src = np.repeat(np.arange(n), deg)
    tgt = rng.integers(0, np.maximum(src, 1))  # below the source: everything could go
    return gg.Graph(off.astype(np.uint32), tgt.astype(np.uint32))


@pytest.mark.parametrize("n,degrees,away", [
    (700, [511, 512, 513, 2047, 2048, 2049], 0.5), (40_000, [513, 1, 2], 0.98),
    ((1 << 21) - 1, [3, 0, 1, 40], 0.7), (1 << 21, [3, 0, 1, 40], 0.7),
    ((1 << 21) + 33, [3, 0, 1, 40], 0.7)])
def test_against_the_oracle(n, degrees, away):
    import paper_2107_12720_gb300 as P
    g = _graph(n, degrees, n)
    mask = (np.random.default_rng(1).random(n) < away).astype(np.uint8)
    with P.Trimmer(g.off, g.tgt) as t:
        t.set_dead_mask(mask)
        for v in ("ac4", "ac6"):
            check_masked(t, g, mask, t.run(v), f"{n} {v}")


def test_long_rows_use_all_sms():
    """16 million look-ups of 20,000 vertices: 34 us, 240 with neighbouring blocks of 32
    vertices on the same SM."""
    import paper_2107_12720_gb300 as P
    n, d = 20_000, 800
    rng = np.random.default_rng(2)
    off = (np.arange(n + 1) * d).astype(np.uint32)
    tgt = rng.integers(0, n, n * d).astype(np.uint32)
    with P.Trimmer(off, tgt) as t:
        t.set_dead_mask((rng.random(n) < 0.5).astype(np.uint8))
        assert min(t.run("ac4")["device_ms"] for _ in range(20)) < 0.12
