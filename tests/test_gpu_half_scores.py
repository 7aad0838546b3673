"""The 16-bit score kernels' fp16 add of gap_open: score bounds at and around
the largest it is used for (2047 + gap_open), saturated scores, ties and
several scorings, bit-exact against the oracle with and without a CIGAR."""
import numpy as np
import pytest

import synth
from gpu_helpers import assert_parity, run_gpu

pytestmark = pytest.mark.gpu


def _batch(reads, wins):
    off = lambda a: np.concatenate([[0], np.cumsum([len(x) for x in a])]).astype(np.int64)  # noqa: E731
    n = len(reads)
    return synth.Workload("bounds", np.concatenate(reads), off(reads), np.concatenate(wins), off(wins),
                          np.arange(n, dtype=np.int64), np.arange(n + 1, dtype=np.int64), np.zeros(n, np.uint8),
                          np.zeros(n, np.int32))


@pytest.mark.parametrize("scoring", [(5, -4, -10, -1), (2, -3, -5, -2), (1, -4, -7, -1), (127 - 14, 0, -14, 0),
                                     (5, -4, -12, -1), (5, -12, -10, -1)])
@pytest.mark.parametrize("cigar", [False, True])
def test_bounds_of_the_fp16_add(scoring, cigar):
    top = (2047 + scoring[2]) // scoring[0]   # longest exact match whose cells stay within 2047
    rng = np.random.default_rng(23)
    reads, wins = [], []
    for m in sorted({17, 60, 101, 103, max(1, top - 1), top, top + 1, top + 2, top + 40}):
        if m > 2100:
            continue
        for alphabet, plant in ((4, True), (4, False), (2, True), (2, False)):
            r = rng.integers(0, alphabet, m).astype(np.uint8)
            w = rng.integers(0, alphabet, m + 90).astype(np.uint8)
            if plant:
                w[30:30 + m] = r
                if alphabet == 2:
                    w = np.concatenate([w[:30 + m // 2], w[31 + m // 2:]])
            reads.append(r)
            wins.append(w)
            reads.append(r)       # the window bounds the score
            wins.append(w[:max(1, m - 1)])
    wl = _batch(reads, wins)
    assert_parity(wl, run_gpu(wl, scoring, cigar=cigar), scoring, cigar=cigar)
