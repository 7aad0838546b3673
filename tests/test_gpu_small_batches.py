"""Batches on both sides of the small-batch limit (4,096 pairs): the few
launches of a small batch and the general sequence give the oracle's scores,
end cells and CIGARs, for mixed lengths (several classes, row chunks and
arithmetic modes), masked and empty pairs, plans and captured calls."""
import numpy as np
import pytest

import synth
from gpu_helpers import assert_parity, run_gpu

pytestmark = pytest.mark.gpu

DEFAULT = (5, -4, -10, -1)


def _mixed(n, rng):
    """n pairs of uneven lengths, among them a 6,500-base read (32-bit cells)
    and reads of several row chunks."""
    wl = synth.generate("uneven", seed=int(rng.integers(1 << 30)), n_reads=max(1, n - 3))
    reads = [wl.reads[a:b] for a, b in zip(wl.read_offsets, wl.read_offsets[1:])]
    wins = [wl.windows[a:b] for a, b in zip(wl.window_offsets, wl.window_offsets[1:])]
    for m in (6500, 2100, 1)[:max(0, n - 1)]:
        r = rng.integers(0, 4, m).astype(np.uint8)
        reads.append(r)
        wins.append(np.concatenate([rng.integers(0, 4, 9).astype(np.uint8), r[:m // 2], r[m // 2 + m // 400:]]))
    off = lambda a: np.concatenate([[0], np.cumsum([len(x) for x in a])]).astype(np.int64)  # noqa: E731
    k = len(reads)
    return synth.Workload("mixed", np.concatenate(reads), off(reads), np.concatenate(wins), off(wins),
                          np.arange(k, dtype=np.int64), np.arange(k + 1, dtype=np.int64), np.zeros(k, np.uint8),
                          np.zeros(k, np.int32))


@pytest.mark.parametrize("n", [1, 2, 33, 1000, 4095, 4096, 4097])
@pytest.mark.parametrize("cigar", [False, True])
def test_both_sides_of_the_limit(n, cigar):
    rng = np.random.default_rng(n)
    wl = _mixed(n, rng)
    got = run_gpu(wl, DEFAULT, cigar=cigar)
    pick = np.unique(np.concatenate([np.arange(max(0, wl.n_pairs - 3), wl.n_pairs),
                                     rng.choice(wl.n_pairs, min(wl.n_pairs, 250), replace=False)]))
    assert_parity(wl, got, DEFAULT, pairs=pick, cigar=cigar)


@pytest.mark.parametrize("m", [513, 601, 640, 801, 1000, 1024, 1601, 2048])
def test_plans_of_20_and_32_rows(m):
    """Reads whose plan has 20 or 32 rows per lane, in one row chunk and in two,
    in a small batch of too many pairs for block tasks."""
    wl = synth.random_pairs(700, (m - 20, m), (m - 10, m + 90), seed=m, alphabet=3)
    for cigar in (False, True):
        got = run_gpu(wl, DEFAULT, cigar=cigar)
        pick = np.sort(np.random.default_rng(m).choice(wl.n_pairs, 40, replace=False))
        assert_parity(wl, got, DEFAULT, pairs=pick, cigar=cigar)


@pytest.mark.parametrize("n", [300, 6000])
def test_masked_and_empty_pairs(n):
    """Unselected pairs and empty windows are finished by the classification
    of either sequence."""
    import torch
    from paper_1304_0681_gb300 import DeviceBatch, _swgb
    rng = np.random.default_rng(n)
    wl = synth.random_pairs(n, (20, 180), (0, 260), seed=n)
    mask = (rng.random(n) < 0.6).astype(np.uint8)
    b = DeviceBatch.from_packed(wl.packed_reads(), wl.read_offsets, wl.packed_windows(), wl.window_offsets,
                                pair_read=wl.pair_read)
    _swgb.sw_batch_align_masked(b.reads, b.read_offsets, b.n_reads, b.windows, b.window_offsets, b.pair_read,
                                torch.from_numpy(mask).cuda(), n, DEFAULT, b.score, b.end, b.cigar_tuple())
    _swgb.sw_sync_status()
    full = run_gpu(wl, DEFAULT)
    score, end, n_ops = b.score.cpu().numpy(), b.end.cpu().numpy().reshape(-1, 2), b.cigar_n.cpu().numpy()
    on = mask != 0
    assert np.array_equal(score[on], full["score"][on]) and np.array_equal(n_ops[on], full["n_ops"][on])
    assert np.array_equal(end[on, 0], full["i_end"][on]) and np.array_equal(end[on, 1], full["j_end"][on])
    assert (score[~on] == -1).all() and (end[~on] == -1).all() and (n_ops[~on] == 0).all()
    assert_parity(wl, full, DEFAULT, pairs=np.sort(rng.choice(n, 200, replace=False)))


def test_a_small_plan_checks_its_shape_and_replays():
    """A planned small batch in a captured graph: replays follow new bases, and
    offsets that no longer fit the plan are reported."""
    import torch
    from paper_1304_0681_gb300 import BatchPlan, DeviceBatch, SwError
    rng = np.random.default_rng(5)
    wl = _mixed(500, rng)
    b = DeviceBatch.from_packed(wl.packed_reads(), wl.read_offsets, wl.packed_windows(), wl.window_offsets)
    plan = BatchPlan(b, DEFAULT)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        plan.align(s)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            plan.align(s)
    flip = synth.pack(((wl.windows + rng.integers(1, 4, len(wl.windows)) * (rng.random(len(wl.windows)) < 0.02)) & 3)
                      .astype(np.uint8))
    b.windows.copy_(torch.from_numpy(flip).cuda())
    graph.replay()
    torch.cuda.synchronize()
    plan.status(s)
    wl.windows = synth.unpack(flip, len(wl.windows))
    end = b.end.cpu().numpy().reshape(-1, 2)
    got = {"score": b.score.cpu().numpy().astype(np.int64), "i_end": end[:, 0], "j_end": end[:, 1],
           "ops": b.cigar_ops.cpu().numpy().view(np.uint32), "cigar_offsets": b.cigar_offsets.cpu().numpy(),
           "n_ops": b.cigar_n.cpu().numpy()}
    assert_parity(wl, got, DEFAULT, pairs=np.sort(rng.choice(wl.n_pairs, 150, replace=False)))
    b.window_offsets[-2] -= 1    # the last window, the longest of its class, grows
    plan.align()
    with pytest.raises(SwError):
        plan.status()
    plan.close()


def test_block_tasks_rows_come_with_the_first_small_batch():
    """A stream of larger batches holds no boundary rows of block tasks (64 MB);
    a small batch captured there runs without them, and the first one outside a
    capture brings them."""
    import torch
    from paper_1304_0681_gb300 import DeviceBatch, align
    s = torch.cuda.Stream()

    def batch(wl, cigar):
        return DeviceBatch.from_packed(wl.packed_reads(), wl.read_offsets, wl.packed_windows(), wl.window_offsets,
                                       cigar=cigar)

    large = batch(synth.random_pairs(5000, (90, 100), (150, 160), seed=1), False)
    wl = synth.random_pairs(24, (600, 2000), (700, 2100), seed=3, alphabet=3)
    small = batch(wl, False)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    align(large, DEFAULT, cigar=False, stream=s)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 100 << 20

    def check(run):
        small.score.fill_(-7)
        small.end.fill_(-7)
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        end = small.end.cpu().numpy().reshape(-1, 2).astype(np.int64)
        got = {"score": small.score.cpu().numpy().astype(np.int64), "i_end": end[:, 0], "j_end": end[:, 1]}
        assert_parity(wl, got, DEFAULT, cigar=False)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        align(small, DEFAULT, cigar=False, stream=s, sync=False)
    check(graph.replay)
    check(lambda: align(small, DEFAULT, cigar=False, stream=s))
    check(graph.replay)
