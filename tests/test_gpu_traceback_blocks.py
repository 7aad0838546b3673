"""The 16-bit traceback recomputes a read in blocks of 50, 60 or 64 rows (by the
score plan's rows per lane) from the score pass's checkpoints: reads whose
length, end row, gaps or start fall on and around the block edges under every
plan, windows on both sides of the wide-window split, every number of lanes per
two pairs, and several scorings, bit-exact against the oracle."""
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


def _edge_pairs(rng, lengths, alphabet=4):
    """Reads with one gap run that begins, ends or lies across a block edge,
    flanked by random bases; some with their first rows unrelated."""
    out = []
    base = lambda n: rng.integers(0, alphabet, n).astype(np.uint8)  # noqa: E731
    for m in lengths:
        for at in sorted({1, m // 2} | {e + d for e in (50, 60, 64, 100, 120, 128) for d in (-1, 0, 1) if 0 < e + d < m - 1}):
            read = base(m)
            for gap in (0, 1, 7, -1, -6, 40, 300):
                if gap >= 0:   # window bases the read lacks
                    win = np.concatenate([read[:at], base(gap), read[at:]])
                else:          # read bases the window lacks
                    win = np.concatenate([read[:at], read[min(m, at - gap):]])
                if rng.random() < 0.3:
                    win = np.concatenate([base(at), win[at:]])   # the alignment starts inside the read
                out.append((read, np.concatenate([base(rng.integers(0, 30)), win, base(rng.integers(0, 30))])))
    return out


EDGES = (39, 40, 41, 49, 50, 51, 59, 60, 61, 63, 64, 65, 81, 101, 121, 129, 151)


@pytest.mark.parametrize("scoring", [DEFAULT, (2, -3, -5, -2), (2, -9, -4, -1), (5, -4, -10, 0), (1, -1, -2, -2)])
def test_gaps_around_block_edges(scoring):
    rng = np.random.default_rng(17)
    wl = _batch(_edge_pairs(rng, EDGES) + _edge_pairs(rng, (66, 102), alphabet=2))
    assert_parity(wl, run_gpu(wl, scoring), scoring)


@pytest.mark.parametrize("rows,block", [(8, 64), (16, 64), (20, 60), (25, 50), (32, 64), (50, 50)])
def test_every_block_height_at_its_edges(rows, block):
    """Each rows-per-lane choice for every read: blocks of its height."""
    import paper_1304_0681_gb300 as sw
    rng = np.random.default_rng(rows)
    lengths = sorted({e + d for e in (block, 2 * block) for d in (-1, 0, 1)} | {block + 20, 2 * block + 23})
    wl = _batch(_edge_pairs(rng, lengths) + _edge_pairs(rng, (block + 1,), alphabet=2))
    sw.sw_set_plan(160, -(-160 // rows), rows)
    try:
        for scoring in (DEFAULT, (2, -3, -5, -2)):
            assert_parity(wl, run_gpu(wl, scoring), scoring)
    finally:
        sw.sw_set_plan(0, 1, 8)


def test_long_reads_and_wide_windows():
    """Several row chunks per pair, and blocks whose band is as wide as an
    intron (competing alignments on both sides of it)."""
    rng = np.random.default_rng(18)
    pairs = []
    for m in (700, 1601, 3300):
        for cut, intron in ((m // 2, 250), (m // 3, 900), (50, 2000)):
            r = rng.integers(0, 4, m).astype(np.uint8)
            w = np.concatenate([r[:cut], rng.integers(0, 4, intron).astype(np.uint8), r[cut:]])
            flip = rng.random(len(w)) < 0.02
            w = np.where(flip, (w + rng.integers(1, 4, len(w))) & 3, w).astype(np.uint8)
            pairs += [(r, w), (r, np.concatenate([w, w[:200]]))]
    wl = _batch(pairs)
    assert_parity(wl, run_gpu(wl, DEFAULT), DEFAULT)


@pytest.mark.parametrize("n_pairs", [500, 12_000, 45_000, 120_000, 400_000])
def test_lanes_per_pair(n_pairs):
    """16, 8, 4, 2 and 1 lanes per two pairs (chosen by the batch's size)."""
    wl = synth.random_pairs(n_pairs, (30, 130), (20, 190), seed=n_pairs, alphabet=3)
    got = run_gpu(wl, DEFAULT)
    sample = np.random.default_rng(3).choice(n_pairs, 500, replace=False)
    assert_parity(wl, got, DEFAULT, pairs=np.sort(sample))


def test_block_doubling_when_the_pool_is_small():
    """More checkpoint rows than the scratch of a batch this size holds: the
    blocks double until they fit."""
    rng = np.random.default_rng(19)
    pairs = []
    for _ in range(40):
        r = rng.integers(0, 4, 6000).astype(np.uint8)
        w = np.concatenate([rng.integers(0, 4, 14_000).astype(np.uint8), r])
        flip = rng.random(len(w)) < 0.02
        pairs.append((r, np.where(flip, (w + rng.integers(1, 4, len(w))) & 3, w).astype(np.uint8)))
    wl = _batch(pairs)
    assert_parity(wl, run_gpu(wl, DEFAULT), DEFAULT, pairs=np.arange(0, 40, 8))


def test_32_bit_pairs_have_all_of_the_scratch():
    """An 8,192-base read that matches with its last 200 bases only: its band
    takes most of a small batch's scratch, which the row checkpoints of the other
    pairs fill before.  Both fit, one after the other."""
    from paper_1304_0681_gb300 import DeviceBatch, _swgb, align
    rng = np.random.default_rng(20)
    r = rng.integers(0, 4, 8192).astype(np.uint8)
    w = np.concatenate([rng.integers(0, 4, 45_000).astype(np.uint8), r[-200:]])
    pairs = [(r, w)]
    for _ in range(70):
        r = rng.integers(0, 4, 6000).astype(np.uint8)
        pairs.append((r, np.concatenate([rng.integers(0, 4, 8000).astype(np.uint8), r])))
    got = []
    for wl in (_batch(pairs[:1]), _batch(pairs)):
        b = DeviceBatch.from_packed(wl.packed_reads(), wl.read_offsets, wl.packed_windows(), wl.window_offsets)
        align(b, DEFAULT)
        _swgb.sw_sync_status()
        n = b.cigar_n.cpu().numpy()
        got.append((int(b.score[0]), b.end[:2].tolist(), b.cigar_ops[:n[0]].tolist()))
        score, ops = b.score.cpu().numpy(), b.cigar_ops.cpu().numpy().view(np.uint32)
    assert got[0] == got[1] and got[0][0] >= 1000
    # the others: exact copies, one run of 6,000 bases
    assert (score[1:] == 30_000).all() and (n[1:] == 1).all()
    assert (ops[b.cigar_offsets.cpu().numpy()[1:-1]] == 6000 << 4).all()
