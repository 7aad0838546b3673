"""A few long reads: the row chunks of two pairs go to the warps of one block,
each a wavefront behind the other.  Read lengths on the edges of the chunk
counts (256, 1024, 2048 and 3200 rows and beyond, where a warp takes several
chunks), windows of one to a few thousand columns, and the batches on the other
side of the rule (too many tasks, rows that do not fit the scratch), bit-exact
against the oracle."""
import numpy as np
import pytest

import synth
from gpu_helpers import assert_parity, run_gpu

pytestmark = pytest.mark.gpu

DEFAULT = (5, -4, -10, -1)


def _batch(pairs):
    reads, wins = zip(*pairs)
    off = lambda a: np.concatenate([[0], np.cumsum([len(x) for x in a])]).astype(np.int64)  # noqa: E731
    n = len(reads)
    return synth.Workload("blocks", np.concatenate(reads), off(reads), np.concatenate(wins), off(wins),
                          np.arange(n, dtype=np.int64), np.arange(n + 1, dtype=np.int64), np.zeros(n, np.uint8),
                          np.zeros(n, np.int32))


def _pair(rng, m, n, like=0.05):
    """A read of m bases and n window columns taken from it with errors, or
    random (n is what the read's copy is cut or padded to)."""
    r = rng.integers(0, 4, m).astype(np.uint8)
    w = np.concatenate([rng.integers(0, 4, 11).astype(np.uint8), r[:m // 3], r[m // 3 + 3:]])
    w = np.where(rng.random(len(w)) < like, (w + 1) & 3, w).astype(np.uint8)
    return r, np.concatenate([w, rng.integers(0, 4, max(0, n - len(w))).astype(np.uint8)])[:n]


@pytest.mark.parametrize("scoring", [DEFAULT, (2, -9, -4, -1), (1, -1, -2, -2)])
@pytest.mark.parametrize("cigar", [False, True])
def test_edges_of_the_chunk_counts(scoring, cigar):
    rng = np.random.default_rng(7)
    pairs = []
    for m in (256, 257, 289, 511, 513, 1023, 1024, 1025, 2047, 2049, 3199, 3201, 4100, 6390):
        for n in (1, 2, 15, 17, 63, 66, m - 1, m + 130):
            pairs.append(_pair(rng, m, n))
        pairs.append(_pair(rng, m, m + 301, like=1.0))
    wl = _batch(pairs)
    assert_parity(wl, run_gpu(wl, scoring, cigar=cigar), scoring, cigar=cigar)


@pytest.mark.parametrize("n_pairs,m,n", [(1216, 300, 410), (1218, 300, 410), (600, 260, 15_000), (7, 600, 9000)])
def test_both_sides_of_the_rule(n_pairs, m, n):
    rng = np.random.default_rng(n_pairs)
    wl = _batch([_pair(rng, m - (i % 3), n + i % 2) for i in range(n_pairs)])
    pick = np.sort(rng.choice(n_pairs, min(n_pairs, 60), replace=False))
    assert_parity(wl, run_gpu(wl, DEFAULT), DEFAULT, pairs=pick)
