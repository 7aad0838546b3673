"""A few long reads: the row chunks of two pairs go to the warps of one block,
each a wavefront behind the other.  Read lengths on the edges of the chunk
counts (from 513 on; 1024, 2048 and 3200 rows and beyond, where a warp takes
several chunks), windows of one to a few thousand columns, and batches on both
sides of the rule's limits (its arithmetic is checked on the host), bit-exact
against the oracle or the general sequence, which has no block tasks."""
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
    for m in (511, 512, 513, 767, 769, 1023, 1024, 1025, 2047, 2049, 3199, 3201, 4100, 6390):
        for n in (1, 2, 15, 17, 63, 66, m - 1, m + 130):
            pairs.append(_pair(rng, m, n))
        pairs.append(_pair(rng, m, m + 301, like=1.0))
    wl = _batch(pairs)
    assert_parity(wl, run_gpu(wl, scoring, cigar=cigar), scoring, cigar=cigar)


def _general(wl, cigar=True):
    """The batch through the general sequence: with any plan override set, here
    one that covers no read, a batch does not take the small launches."""
    import paper_1304_0681_gb300 as sw
    sw.sw_set_plan(1, 1, 8)
    try:
        return run_gpu(wl, DEFAULT, cigar=cigar)
    finally:
        sw.sw_set_plan(0, 1, 8)


def _same(wl, a, b):
    for k in ("score", "i_end", "j_end"):
        assert np.array_equal(a[k], b[k])
    if "ops" in a:
        assert np.array_equal(a["n_ops"], b["n_ops"])
        for p in range(wl.n_pairs):
            o, n = a["cigar_offsets"][p], a["n_ops"][p]
            assert np.array_equal(a["ops"][o:o + n], b["ops"][o:o + n])


@pytest.mark.parametrize("tasks_over", [-1, 0, 1])
@pytest.mark.parametrize("m,n", [(600, 650), (1100, 900)])
def test_as_many_tasks_as_blocks(tasks_over, m, n):
    """One task of two pairs per block of the score launch (255 registers: two
    blocks of 128 threads per SM), one fewer, and one more than that."""
    import torch
    tasks = 2 * torch.cuda.get_device_properties(0).multi_processor_count + tasks_over
    rng = np.random.default_rng(m + tasks)
    wl = _batch([_pair(rng, m - (i % 3), n + i % 2) for i in range(2 * tasks - 1)])
    got = run_gpu(wl, DEFAULT)
    _same(wl, got, _general(wl))
    assert_parity(wl, got, DEFAULT, pairs=np.sort(rng.choice(wl.n_pairs, 60, replace=False)))


@pytest.mark.parametrize("lengths,pairs,n", [
    ((600,), 12, 9000),                   # well inside
    ((600, 700, 1100), 32, 120_000),      # three classes of 30.7 MB of rows: two find room
    ((650,), 72, 120_000),                # one class of 69 MB: none
])
def test_rows_within_and_past_the_scratch(lengths, pairs, n):
    """The boundary rows of all block tasks share 64 MB; a class that finds no
    room runs as warp tasks, beside classes that did."""
    rng = np.random.default_rng(n + pairs)
    out = []
    for m in lengths:
        for _ in range(pairs):
            r = rng.integers(0, 4, m).astype(np.uint8)
            w = rng.integers(0, 4, n).astype(np.uint8)
            at = int(rng.integers(0, n - m))
            w[at:at + m] = np.where(rng.random(m) < 0.03, (r + 1) & 3, r)
            out.append((r, w))
    wl = _batch(out)
    got = run_gpu(wl, DEFAULT, cigar=False)
    _same(wl, got, _general(wl, cigar=False))
    if n < 10_000:
        assert_parity(wl, got, DEFAULT, cigar=False)
