"""G^T built on the device where its sort changes form, against the oracle's
transpose: edge counts around a tile (16,384) and around the pieces of the CTAs,
rows longer than several tiles, long runs of empty rows, all edges in one bucket
(too large for shared memory) or in one target, and vertex counts around the number
of buckets."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def csr(src, dst, n):
    order = np.argsort(src, kind="stable")
    off = np.zeros(n + 1, np.uint32)
    np.cumsum(np.bincount(src, minlength=n), out=off[1:])
    return gg.Graph(off, dst[order].astype(np.uint32), name="csr")


def uniform(n, m, seed):
    rng = np.random.default_rng(seed)
    return csr(rng.integers(0, n, m), rng.integers(0, n, m), n)


def long_rows(n, m, rows):
    rng = np.random.default_rng(m)
    return csr(rng.choice(np.linspace(0, n - 1, rows).astype(np.int64), m),
               rng.integers(0, n, m), n)


def narrow_targets(n, m, targets):
    rng = np.random.default_rng(m + targets)
    return csr(rng.integers(0, n, m), n - 1 - rng.integers(0, targets, m), n)


CASES = {
    "one edge": lambda: csr(np.array([2]), np.array([0]), 3),
    "fewer edges than CTAs": lambda: uniform(50, 100, 1),
    **{f"edges {m}": (lambda m=m: uniform(5_000, m, m)) for m in (16_383, 16_384, 16_385)},
    **{f"vertices {n}": (lambda n=n: uniform(n, 60_000, n)) for n in (255, 256, 257, 4095, 4097)},
    "pieces of a tile and a bit": lambda: uniform(70_001, 152 * 16_384 + 300_000, 3),
    "three rows": lambda: long_rows(100_000, 3_000_000, 3),
    "empty rows": lambda: long_rows(2_000_003, 500_000, 700),
    "one target": lambda: narrow_targets(40_000, 1_000_000, 1),
    "one bucket": lambda: narrow_targets(1 << 16, 4_000_000, 100),
    "few buckets": lambda: narrow_targets(1 << 20, 6_000_000, 9_000),
}


@pytest.mark.parametrize("name", list(CASES))
def test_against_the_oracle(name):
    import paper_2107_12720_gb300 as P
    g = CASES[name]()
    want_off, want_tgt = oracle.transpose(g.off, g.tgt)
    with P.Trimmer(g.off, g.tgt) as t:
        got_off, got_tgt = t.in_csr()
    assert np.array_equal(got_off, want_off)
    row = np.repeat(np.arange(want_off.size - 1), np.diff(want_off.astype(np.int64)))
    order = np.lexsort((got_tgt, row))  # the order within a row is unspecified
    assert np.array_equal(got_tgt[order], want_tgt)
