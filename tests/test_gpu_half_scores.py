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


def test_long_reads_of_three_modes_share_the_boundary_scratch():
    """A 1,700-base read on a short window has scores the fp16 add could take,
    but runs in row chunks: a launch of its own would take a third part of the
    boundary rows' scratch, and the rows of the two 700,000-base windows, at
    most half of it each, would no longer fit theirs."""
    import torch
    from paper_1304_0681_gb300 import DeviceBatch, _swgb, align
    rng = np.random.default_rng(31)
    reads = [rng.integers(0, 4, 40).astype(np.uint8) for _ in range(4100)]
    wins = [rng.integers(0, 4, 60).astype(np.uint8) for _ in range(4100)]
    r = rng.integers(0, 4, 1700).astype(np.uint8)
    reads.append(r)
    wins.append(r[200:500].copy())
    for m in (2000, 6500):     # 16-bit cells and 32-bit cells; the read's copy starts at column 1000
        r = rng.integers(0, 4, m).astype(np.uint8)
        w = rng.integers(0, 4, 700_000).astype(np.uint8)
        w[1000:1000 + m] = r
        reads.append(r)
        wins.append(w)
    wl = _batch(reads, wins)
    b = DeviceBatch.from_packed(wl.packed_reads(), wl.read_offsets, wl.packed_windows(), wl.window_offsets, cigar=False)
    align(b, (5, -4, -10, -1), cigar=False)
    _swgb.sw_sync_status()
    end = b.end.cpu().numpy().reshape(-1, 2).astype(np.int64)
    score = b.score.cpu().numpy().astype(np.int64)
    torch.cuda.synchronize()
    assert score[-2:].tolist() == [5 * 2000, 5 * 6500]
    assert end[-2:].tolist() == [[1999, 2999], [6499, 7499]]
    assert_parity(wl, {"score": score, "i_end": end[:, 0], "j_end": end[:, 1]}, (5, -4, -10, -1),
                  pairs=np.arange(4000, 4101), cigar=False)
