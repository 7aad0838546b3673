"""The work that users of this framework have it do, as measurable cases.

A case is one call (or the few calls that belong together) through the
public entry points: a batch aligned on the device, a planned batch, a batch
in host memory, the best hit of every read over its candidates (exhaustive
and filtered), the filter network's forward pass and training step, and a
whole map of reads onto a reference.  Inputs are synthetic and made on the GPU
from a seed: reads of uniform bases, windows that hold the mutated read
between random flanks, paralog-like and random decoys, spliced windows.
"""
import math

import torch

from paper_1304_0681_gb300 import BatchPlan, DeviceBatch, KmerIndex, SeedParams, align, map_reads
from paper_1304_0681_gb300 import filter as flt
from paper_1304_0681_gb300 import sw_batch_align_host_dense, sw_packed_bytes

SCORING = (5, -4, -10, -1)   # match, mismatch, gap open, gap extend
# read lengths and shares of an uneven batch (Illumina runs of several kinds)
MIXED = ((75, .20), (100, .30), (150, .25), (250, .15), (400, .07), (800, .03))
# selection rules of a filtered search: (longest read, k, tau, delta)
RULES = [(112, 4, 0.0, 0.15), (160, 3, 0.0, 0.12), (320, 3, 0.0, 0.1), (448, 2, 0.0, 0.08),
         (2 ** 31 - 1, 1, 0.0, 0.04)]
N_PAR = 33153                # parameters of the filter network


def listed():
    return [
        # a handful of candidate pairs aligned as they come: latency
        dict(name="pairs_64", kind="align", reads=64, length=100, window=150, decoys=0.0, splice=0.0),
        # a small batch of short reads, alignment and CIGAR
        dict(name="pairs_1k", kind="align", reads=1000, length=100, window=150, decoys=0.0, splice=0.0),
        # the same batch shape again and again through a plan, as a service with a fixed batch does
        dict(name="plan_16k", kind="plan", reads=16384, length=100, window=200, decoys=0.2, splice=0.0),
        # the throughput batch: one length, a fifth of the windows without a true match
        dict(name="pairs_1M", kind="align", reads=1_000_000, length=100, window=200, decoys=0.2, splice=0.0),
        # an RNA batch of uneven reads, a tenth of them across an intron
        dict(name="uneven_2M", kind="align", reads=2_000_000, length=0, window=0, decoys=0.0, splice=0.10),
        # long reads of uneven length: several row chunks per pair
        dict(name="long_200", kind="align", reads=200, length=-4000, window=0, decoys=0.0, splice=0.05),
        # a batch in host memory, results and dense CIGARs back on the host
        dict(name="host_200k", kind="host", reads=200_000, length=150, window=250, decoys=0.1, splice=0.0),
        # every candidate of every read aligned, best hit per read (score and end only)
        dict(name="exhaustive_30k", kind="exhaustive", reads=30_000, cands=64, length=150, window=250, splice=0.0),
        # the filtered search on a full mix of reads: features, network, selection, alignment of the selected
        dict(name="filtered_200k", kind="filtered", reads=200_000, cands=32, length=0, window=0, splice=0.15),
        # predictions for the candidates of a batch whose features are in hand
        dict(name="predict_2M", kind="predict", rows=2_000_000),
        # one training step of the filter network (gradient and Adam) on a minibatch
        dict(name="train_4096", kind="train", rows=200_000, batch=4096),
        # reads mapped onto a reference: seeds, windows, alignment with CIGAR, records, top hits
        dict(name="map_200k", kind="map", reads=200_000, length=100, bases=64_000_000, k=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _drawn(rng)
    while work(case)["flops"] > 1e12:   # no more than the largest listed case
        case["reads"] //= 2
    return case


def _drawn(rng):
    kind = rng.choice(["align", "align", "align", "align", "plan", "host", "exhaustive", "filtered", "predict",
                       "train", "map"])
    if kind in ("align", "plan", "host"):
        length = rng.choice([0, 0, rng.randint(50, 420), rng.randint(50, 420), rng.choice([75, 100, 150, 250, 400]),
                             rng.randint(600, 1500), -rng.randint(1500, 8000)])
        longest = 100_000_000 if kind != "host" else 30_000_000       # read bases
        n = _log(rng, 32, max(64, min(600_000, longest // max(160, abs(length)))))
        if length < 0:   # up to the longest reads the library takes (32-bit cells past 6,400 bases)
            n = min(n, int(2e9 / length ** 2))
        window = length + rng.randint(30, 120) if length > 0 and rng.random() < 0.5 else 0
        return dict(kind=kind, reads=n, length=length, window=window, decoys=rng.choice([0.0, 0.1, 0.3]),
                    splice=rng.choice([0.0, 0.0, 0.1, 0.2]) if not window else 0.0)
    if kind in ("exhaustive", "filtered"):
        length = rng.choice([0, rng.randint(60, 420), 100, 150])
        return dict(kind=kind, reads=_log(rng, 50, 100_000), cands=rng.choice([4, 16, 32, 64]), length=length,
                    window=length + rng.randint(30, 120) if length and rng.random() < 0.5 else 0,
                    splice=rng.choice([0.0, 0.15]))
    if kind == "predict":
        return dict(kind=kind, rows=_log(rng, 500, 4_000_000))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 10_000, 500_000), batch=_log(rng, 256, 8192))
    return dict(kind=kind, reads=_log(rng, 500, 300_000), length=rng.choice([75, 100, 150, 250]),
                bases=_log(rng, 2_000_000, 64_000_000), k=rng.choice([11, 12, 13]))


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & (2 ** 62 - 1))
    return g


def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda")


def _ints(g, lo, hi, n, dtype=torch.int64):
    return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=dtype)


def _offsets(lengths):
    off = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device=lengths.device)
    torch.cumsum(lengths, 0, out=off[1:])
    return off


def _pack(codes):
    """2-bit packing, four bases per byte, the first in the low bits."""
    n = codes.numel()
    buf = torch.zeros(4 * sw_packed_bytes(n), dtype=torch.uint8, device=codes.device)
    buf[:n] = codes
    q = buf.view(-1, 4)
    return q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)


def _read_lengths(g, case):
    n, length = case["reads"], case["length"]
    if length > 0:
        return torch.full((n,), length, dtype=torch.int64, device="cuda")
    at = (torch.randperm(n, generator=g, device="cuda").double() + 0.5) / n
    if length < 0:   # long reads: evenly from a quarter of -length up to it
        return (-length * (0.25 + 0.75 * at)).to(torch.int64)
    share = torch.tensor([w for _, w in MIXED], dtype=torch.float64, device="cuda").cumsum(0)
    share[-1] = 1.0
    return torch.tensor([v for v, _ in MIXED], dtype=torch.int64, device="cuda")[torch.searchsorted(share, at)]


def _fill_windows(g, reads, rs, m, copied, div, spliced, window):
    """Windows of one group of pairs: codes back to back, and their lengths.
    A pair has m + 2 slots: the left flank, one per read base, the right
    flank; a slot gives any number of window bases."""
    n = m.numel()
    off = _offsets(m + 2)
    total = int(off[-1])
    pid = torch.repeat_interleave(torch.arange(n, device="cuda"), m + 2, output_size=total)
    pos = torch.arange(total, device="cuda") - off[pid] - 1
    mp = m[pid]
    base = (pos >= 0) & (pos < mp)
    event = base & (_rand(g, total) < div[pid])
    kind = _rand(g, total)
    size = _ints(g, 1, 3, total, torch.int32)
    dele = event & (kind > 0.9)
    gone = dele.clone()
    gone[1:] |= dele[:-1] & (size[:-1] >= 2)
    gone[2:] |= dele[:-2] & (size[:-2] >= 3)
    count = torch.where(event & (kind > 0.8) & (kind <= 0.9), 1 + size, 1).to(torch.int64)
    count = torch.where(gone, 0, count)
    cut = base & (pos == mp // 2) & spliced[pid]
    count = torch.where(cut, 1 + _ints(g, 50, 2000, total), count)
    count = torch.where(base, count, 0)
    inner = torch.zeros(total + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(count, 0, out=inner[1:])
    inner = inner[off[1:]] - inner[off[:-1]]
    if window:
        left = (_rand(g, n) * (window - inner + 1).clamp(min=1)).to(torch.int64)
        right = (window - inner - left).clamp(min=0)
    else:
        left, right = _ints(g, 20, 100, n), _ints(g, 20, 100, n)
    count[off[:-1]] = left
    count[off[1:] - 1] = right
    sub = event & (kind <= 0.8)
    code = (reads[(rs[pid] + pos).clamp(0, reads.numel() - 1)] + sub * _ints(g, 1, 3, total, torch.uint8)) & 3
    keep = base & copied[pid]
    del pid, pos, mp, kind, size, dele, gone, event, sub, base
    ends = torch.cumsum(count, 0)
    out = int(ends[-1])
    src = torch.repeat_interleave(torch.arange(total, device="cuda"), count, output_size=out)
    e = torch.arange(out, device="cuda") - (ends - count)[src]
    codes = _ints(g, 0, 3, out, torch.uint8)
    codes = torch.where((e == 0) & keep[src], code[src], codes)
    last = count[src] - e
    intron = cut[src] & keep[src]
    for where, value in ((e == 1, 2), (e == 2, 3), (last == 2, 0), (last == 1, 2)):   # GT ... AG
        codes = torch.where(intron & where, value, codes)
    return codes, inner + left + right


def _workload(case, seed):
    """Reads, windows and offsets on the device; with "cands" every read has
    1 to that many windows, one of them its own."""
    g = _gen(seed)
    rl = _read_lengths(g, case)
    roff = _offsets(rl)
    reads = _ints(g, 0, 3, int(roff[-1]), torch.uint8)
    n = case["reads"]
    cands = case.get("cands", 0)
    if cands:
        nc = 1 + torch.randperm(n, generator=g, device="cuda") % cands
        coff = _offsets(nc)
        pair_read = torch.repeat_interleave(torch.arange(n, device="cuda"), nc)
        rank = torch.arange(pair_read.numel(), device="cuda") - coff[pair_read]
        true = rank == (_rand(g, n) * nc).to(torch.int64)[pair_read]
        u = _rand(g, pair_read.numel())
        copied = true | (_rand(g, pair_read.numel()) < 0.5)   # the rest: random windows
        div = torch.where(true, 0.01 + 0.04 * u, 0.05 + 0.15 * u)
    else:
        coff, pair_read = None, torch.arange(n, device="cuda")
        copied = _rand(g, n) >= case["decoys"]
        div = 0.025 * torch.ones(n, device="cuda") if case["window"] else 0.005 + 0.045 * _rand(g, n)
    spliced = (_rand(g, n) < case["splice"])[pair_read]
    m, rs = rl[pair_read], roff[pair_read]
    codes, lens = [], []
    pairs = max(1, int(48_000_000 / max(1.0, float((m + 2).float().mean()))))
    for p in range(0, m.numel(), pairs):
        q = slice(p, p + pairs)
        c, ln = _fill_windows(g, reads, rs[q], m[q], copied[q], div[q], spliced[q], case["window"])
        codes.append(c)
        lens.append(ln)
    lens = torch.cat(lens)
    return dict(reads=_pack(reads), roff=roff, wins=_pack(torch.cat(codes)), woff=_offsets(lens),
                pair_read=pair_read if cands else None, coff=coff, m=m)


def _batch(w, cigar):
    n = w["m"].numel()
    coff = _offsets(2 * w["m"] + 3) if cigar else None
    new = lambda k: torch.zeros(k, dtype=torch.int32, device="cuda")  # noqa: E731
    return DeviceBatch(w["reads"], w["roff"], w["wins"], w["woff"], w["pair_read"], new(n), new(2 * n),
                       new(int(coff[-1])) if cigar else None, coff, new(n) if cigar else None)


def _model(seed):
    """A network whose prediction ranks as a trained one does: the shared
    4-mers, plus smaller terms of every unit."""
    model = flt.FilterModel(seed=int(seed) & 0xFFFFFFFF)
    p = model.params().clone()
    w1, w2 = p[:16384].view(64, 256), p[16640:33024].view(256, 64)
    w1 *= 0.5
    w1[:, 0] = 1.0
    w2[:, 0] = 0.0
    w2[0, 0] = 1.0
    p[16384:16640] = 0.05 * torch.randn(256, generator=_gen(seed + 1), device="cuda")
    p[33024:33088] = 0.05 * torch.randn(64, generator=_gen(seed + 2), device="cuda")
    p[33088] = 1.0
    p[33152] = 0.0
    model.set_params(p)
    return model


def _feature_rows(seed, n):
    """Shared 4-mer counts over a 97-position read, as the feature kernel gives them."""
    counts = torch.poisson(torch.full((n, 64), 0.7, device="cuda"), generator=_gen(seed))
    return (counts / 97.0).to(torch.bfloat16).view(torch.int16)


def _genome(seed, bases):
    codes = _ints(_gen(seed), 0, 3, bases, torch.uint8)
    return codes, [bases * c // 8 for c in range(9)]


def _sampled_reads(g, codes, n, m):
    """Reads of m bases from either strand, 1% substituted, some with one indel."""
    start = (_rand(g, n) * (codes.numel() - m - 8)).to(torch.int64)
    step = torch.ones(n, m, dtype=torch.int64, device="cuda")
    hit = torch.nonzero(_rand(g, n) < min(0.9, 0.003 * m)).reshape(-1)
    step[hit, _ints(g, 5, m - 6, hit.numel())] = 3 * (_rand(g, hit.numel()) < 0.5).to(torch.int64)
    at = (start[:, None] + torch.cumsum(step, 1)).clamp(max=codes.numel() - 1)
    r = codes[at]
    r = (r + (_rand(g, n * m).view(n, m) < 0.01) * _ints(g, 1, 3, n * m, torch.uint8).view(n, m)) & 3
    back = _rand(g, n) < 0.5
    r = torch.where(back[:, None], 3 - r.flip(1), r)
    return _pack(r.reshape(-1)), torch.arange(n + 1, device="cuda") * m


def _room(n_pairs, slots):
    """CIGAR runs of a batch with room to spare (a run is several bases long on average)."""
    return 8 * n_pairs + slots // 16


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("align", "plan"):
        b = _batch(_workload(case, seed), True)
        s = dict(kind=kind, batch=b, room=_room(b.n_pairs, int(b.cigar_offsets[-1])))
        if b.cigar_ops.numel() <= 4_000_000:   # which pair a CIGAR slot belongs to, and where in its slot it is
            s["slot_pair"] = torch.repeat_interleave(torch.arange(b.n_pairs, device="cuda"),
                                                     b.cigar_offsets[1:] - b.cigar_offsets[:-1])
            s["slot_pos"] = torch.arange(b.cigar_ops.numel(), device="cuda") - b.cigar_offsets[s["slot_pair"]]
        if kind == "plan":
            s["plan"] = BatchPlan(b, SCORING, cigar=True)
        return s
    if kind == "host":
        w = _workload(case, seed)
        n = w["m"].numel()
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        new = lambda k, t: torch.zeros(k, dtype=t).pin_memory()  # noqa: E731
        return dict(kind=kind, n=n, reads=pin(w["reads"]), roff=pin(w["roff"]), wins=pin(w["wins"]),
                    woff=pin(w["woff"]), score=new(n, torch.int32), end=new(2 * n, torch.int32),
                    ops=new(_room(n, int((2 * w["m"] + 3).sum())), torch.int32), offsets=new(n + 1, torch.int64))
    if kind in ("exhaustive", "filtered"):
        w = _workload(case, seed)
        s = dict(kind=kind, batch=_batch(w, False), coff=w["coff"])
        if kind == "filtered":
            s["model"] = _model(3)
        return s
    if kind == "predict":
        return dict(kind=kind, model=_model(seed), x=_feature_rows(seed, case["rows"]))
    if kind == "train":
        n = case["rows"]
        x = _feature_rows(seed, n)
        y = x.view(torch.bfloat16).float().sum(1)
        y = (y * 0.6 + 0.1 * torch.rand(n, generator=_gen(seed + 5), device="cuda")).contiguous()
        idx = _ints(_gen(seed + 6), 0, n - 1, case["batch"], torch.int32)
        return dict(kind=kind, model=_model(seed), x=x, y=y, idx=idx)
    codes, chrom = _genome(seed, case["bases"])
    reads, roff = _sampled_reads(_gen(seed + 7), codes, case["reads"], case["length"])
    index = KmerIndex(_pack(codes), chrom, k=case["k"])
    windows = 4 * case["reads"] + 1024
    return dict(kind="map", index=index, reads=reads, roff=roff, n=case["reads"], params=SeedParams(k=case["k"]),
                min_score=2 * case["length"], windows=windows, room=_room(windows, 0))


# ------------------------------------------------------------------ one pass

def _cigars(s, ops, offsets, n_ops):
    """The CIGAR runs of every pair: a small batch as its slots with the
    unused part cleared, a large one taken out of its slots back to back."""
    if "slot_pair" in s:
        return torch.where(s["slot_pos"] < n_ops[s["slot_pair"]], ops, 0)
    n = n_ops.to(torch.int64)
    first = offsets[:-1] - torch.cumsum(n, 0) + n
    at = torch.repeat_interleave(first, n)
    return _held(ops[at + torch.arange(at.numel(), device=at.device)], s["room"])


def _held(t, room):
    """`t` in a buffer of a size that does not depend on the data."""
    out = torch.zeros((room,) + tuple(t.shape[1:]), dtype=t.dtype, device=t.device)
    out[:t.shape[0]] = t
    return out


def run(s):
    kind = s["kind"]
    if kind in ("align", "plan"):
        b = s["batch"]
        if kind == "plan":
            s["plan"].align()
        else:
            align(b, SCORING)
        return [b.score, b.end, b.cigar_n, _cigars(s, b.cigar_ops, b.cigar_offsets, b.cigar_n)]
    if kind == "host":
        sw_batch_align_host_dense(s["reads"], s["roff"], s["wins"], s["woff"], s["n"], SCORING, s["score"], s["end"],
                                  s["ops"], s["offsets"])
        return [s["score"], s["end"], s["offsets"], s["ops"]]
    if kind == "exhaustive":
        best, cand = flt.exhaustive_best(s["batch"], s["coff"], SCORING)
        return [best, cand, s["batch"].score, s["batch"].end]
    if kind == "filtered":
        r = flt.filtered_best(s["batch"], s["coff"], s["model"], RULES, SCORING)
        return [r.best_score, r.best_cand, r.mask, r.pred, s["batch"].score, s["batch"].end]
    if kind == "predict":
        return s["model"].forward(s["x"])
    if kind == "train":
        m = s["model"]
        m.grad(s["x"], s["y"], s["idx"])
        m.adam(1e-3)
        return [m.gradient(), m.params()]
    mp = map_reads(s["index"], s["reads"], s["roff"], s["n"], SCORING, s["params"], min_score=s["min_score"])
    ops, offsets, n_ops = mp.cigar_tuple()
    w, most = mp.windows, s["windows"]
    return [mp.best_score, mp.best_cand, mp.second_score, mp.mapq, w["cand_offsets"], _held(w["start"], most),
            _held(w["length"], most), _held(mp.score, most), _held(mp.end, 2 * most), _held(n_ops, most),
            _cigars(s, ops, offsets, n_ops), _held(mp.records_dev[:mp.n_records], most)]


# ------------------------------------------------- what a pass cannot do without

def _shape(case):
    """Expected read length, window length and cells of a pair."""
    length, window = case["length"], case["window"]
    if length > 0:
        lens = ((length, 1.0),)
    elif length < 0:
        lens = tuple((-length * (0.25 + 0.75 * (k + 0.5) / 16), 1 / 16) for k in range(16))
    else:
        lens = MIXED
    n = lambda m: window if window else m + 120 + 1025 * case["splice"]  # noqa: E731
    return (sum(w * m for m, w in lens), sum(w * n(m) for m, w in lens), sum(w * m * n(m) for m, w in lens))


def work(case):
    """Bytes of the inputs and outputs, each once; operations: 7 per cell of
    the dynamic program (E, F, diagonal, H, its floor, the substitution and
    the running maximum), two per multiply-add of the network."""
    kind = case["kind"]
    net = 2 * (64 * 256 + 256 * 64 + 64)
    if kind == "predict":
        return {"bytes": case["rows"] * (128 + 4) + 4 * N_PAR, "flops": case["rows"] * net}
    if kind == "train":
        return {"bytes": case["batch"] * (128 + 8) + 4 * N_PAR * 8, "flops": 3 * case["batch"] * net}
    if kind == "map":
        # about one window per read; read, genome span, index buckets, outputs
        n, m = case["reads"], case["length"]
        seeds = 2 * 2 * (m // 12)
        return {"bytes": n * (m / 4 + (m + 90) / 4 + seeds * 32 + 120), "flops": 7 * n * m * (m + 75)}
    m, n, cells = _shape(case)
    pairs = case["reads"] * ((case["cands"] + 1) / 2 if case.get("cands") else 1)
    data = case["reads"] * (m / 4 + 8) + pairs * (n / 4 + 8 + 12)
    if kind == "exhaustive":
        return {"bytes": data + 8 * pairs, "flops": 7 * pairs * cells}
    if kind == "filtered":
        # 4-mer counts, the network, and cells of about a third of the pairs
        return {"bytes": data + 13 * pairs, "flops": pairs * (net + n + 7 * cells / 3)}
    return {"bytes": data + pairs * (4 + 20), "flops": 7 * pairs * cells}


def tolerance(case):
    """Scores, cells, CIGARs, windows and hits are whole numbers and exact.
    The network's numbers carry bf16 operands with fp32 sums."""
    if case["kind"] == "predict":
        return {"rel": 1e-2}
    if case["kind"] == "train":
        return {"rel": 5e-3}
    if case["kind"] == "filtered":
        return {"rel": 1e-2, "differ": 2e-3}   # a rounding of a prediction may change a selection
    return "exact"


def exact(case, seed):
    if case["kind"] not in ("predict", "train"):
        return None
    s = prepare(case, seed)
    p = s["model"].params().double()
    x = s["x"].view(torch.bfloat16)
    w1, b1, w2 = p[:16384].view(64, 256), p[16384:16640], p[16640:33024].view(256, 64)
    b2, w3, b3 = p[33024:33088], p[33088:33152], p[33152]
    if case["kind"] == "predict":
        y = [(torch.relu(torch.relu(c.double() @ w1 + b1) @ w2 + b2) @ w3 + b3) for c in x.split(500_000)]
        return torch.cat(y)
    at = s["idx"].long()
    f, t = x[at].double(), s["y"][at].double()
    z1 = f @ w1 + b1
    a1 = torch.relu(z1)
    z2 = a1 @ w2 + b2
    a2 = torch.relu(z2)
    dy = 2.0 / at.numel() * (a2 @ w3 + b3 - t)
    dz2 = dy[:, None] * w3 * (z2 > 0)
    dz1 = (dz2 @ w2.t()) * (z1 > 0)
    grad = torch.cat([(f.t() @ dz1).reshape(-1), dz1.sum(0), (a1.t() @ dz2).reshape(-1), dz2.sum(0), a2.t() @ dy,
                      dy.sum().reshape(1)])
    # Adam's first step from zero moments
    return [grad, p - 1e-3 * grad / (grad.abs() + 1e-8)]
