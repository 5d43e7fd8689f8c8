"""Performance cases of the k-mer analysis library: what its users run, over the sizes they run
it at. listed() names the cases, draw() gives more of the same ranges, prepare() makes a case's
inputs and handles on the GPU, run() is one pass through the public entry points.

Records come out of the library in unspecified order, so most counting cases read their results
the way an assembler does, by looking k-mers up (the genome's own k-mers in either orientation,
and the same k-mers with one base changed, most of them absent); one orders the records by key.
"""
import math

import numpy as np
import torch

from paper_1705_11147_gb300 import BatchGraph, KmerAnalysis, host_result_buffers, make_params
from paper_1705_11147_gb300.kmer_analysis import estimate_distinct, parse_fastq

MAX_QUERIES = 2_000_000   # genome positions looked up per pass (as many again with a changed base)

COUNT = dict(kind="count", genome=0, coverage=30.0, read_min=150, read_max=150, err=0.01, n_rate=0.0, repeats=0.0,
             satellite=False, k=31, min_depth=2, bloom=True, canonical=True, host=False, records=False)


def listed():
    return [
        # a plasmid or an amplicon panel: the smallest call of a serving loop, one table
        dict(COUNT, name="plasmid_20k", genome=20_000, coverage=25.0, err=0.005),
        # the plain workload of the benchmark: 1 Mbp, 30x of 150 bp, k = 31
        dict(COUNT, name="plain_1m", genome=1_000_000, err=0.005),
        # the bacterial workload: 5 Mbp, 50x, repeats, N bases, two-word keys
        dict(COUNT, name="bacterial_5m", genome=5_000_000, coverage=50.0, n_rate=1e-4, repeats=0.03, k=51),
        # the large-genome workload (30x of 250 bp, 5 % repeats, min depth 4) at half its genome,
        # so that three states fit the card: 3 Gbases
        dict(COUNT, name="large_100m", genome=100_000_000, read_min=250, read_max=250, repeats=0.05, k=51, min_depth=4),
        # quality-trimmed (ragged) reads counted exactly, every k-mer kept, no Bloom filter, and
        # the records taken out and ordered by key (a k-mer database)
        dict(COUNT, name="trimmed_k21", genome=1_500_000, coverage=20.0, read_min=30, read_max=301, err=0.004, k=21, min_depth=1,
             bloom=False, records=True),
        # a repeat-rich genome: 30 % of the reads from a satellite array, heavy hitters expected
        dict(COUNT, name="satellite_10m", genome=10_000_000, satellite=True),
        # reads arrive in pinned host memory and records go back to it, as a pipeline stage runs
        dict(COUNT, name="host_4m", genome=4_000_000, k=51, host=True),
        # many samples of uneven size as one CUDA graph per step
        dict(kind="batch", name="batch_16", samples=16, genome_min=100_000, genome_max=2_000_000, k=51),
        # lookups in a table that stays resident
        dict(kind="query", name="lookup_3m", genome=3_000_000, queries=1_500_000, k=31),
        # the sizing pass before a count: distinct k-mers and heavy hitters
        dict(kind="estimate", name="sizing_3m", genome=3_000_000, coverage=30.0, read_min=150, read_max=150, err=0.01, k=31),
        # FASTQ text to reads: the input side
        dict(kind="fastq", name="fastq_150", bases=100_000_000, read_min=150, read_max=150, crlf=False, host=False),
        # contigs of a finalized sample
        dict(kind="contigs", name="contigs_4m", genome=4_000_000, coverage=30.0, read_min=150, read_max=150, err=0.002, k=51),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count"] * 6 + ["batch", "query", "estimate", "fastq", "contigs"])
    rmin = rng.choice([100, 101, 150, 250, rng.randint(35, 250)])
    rmax = rmin if rng.random() < 0.6 else rmin + rng.randint(1, 120)
    k = rng.choice([21, 25, 31, 31, 33, 51, 51, 63])
    err = round(rng.uniform(0.002, 0.015), 4)
    if kind == "count":
        bloom = rng.random() < 0.8
        genome = _log(rng, 20_000, 40_000_000 if bloom else 3_000_000)
        records = genome < 2_000_000 and rng.random() < 0.2
        return dict(COUNT, genome=genome, coverage=round(rng.uniform(15, 60), 1), read_min=rmin, read_max=rmax, err=err,
                    n_rate=rng.choice([0.0, 1e-4]), repeats=rng.choice([0.0, 0.03]), satellite=rng.random() < 0.1,
                    k=k, min_depth=rng.choice([2, 2, 3, 4]) if bloom else rng.choice([1, 2]), bloom=bloom,
                    canonical=rng.random() < 0.9, host=not records and genome < 8_000_000 and rng.random() < 0.15, records=records)
    if kind == "batch":
        lo = _log(rng, 30_000, 300_000)
        return dict(kind="batch", samples=rng.randint(3, 24), genome_min=lo, genome_max=lo * rng.randint(2, 10), k=k)
    if kind == "query":
        return dict(kind="query", genome=_log(rng, 50_000, 8_000_000), queries=_log(rng, 1_001, 4_000_000), k=k)
    if kind == "estimate":
        return dict(kind="estimate", genome=_log(rng, 30_000, 10_000_000), coverage=round(rng.uniform(10, 40), 1), read_min=rmin,
                    read_max=rmax, err=err, k=k)
    if kind == "fastq":
        return dict(kind="fastq", bases=_log(rng, 200_000, 300_000_000), read_min=rmin, read_max=rmax, crlf=rng.random() < 0.3,
                    host=rng.random() < 0.3)
    return dict(kind="contigs", genome=_log(rng, 50_000, 6_000_000), coverage=round(rng.uniform(20, 40), 1), read_min=max(rmin, 100),
                read_max=max(rmax, 100), err=round(rng.uniform(0.001, 0.004), 4), k=k)


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))


def _randint(lo, hi, n, g, dtype=torch.int64):
    return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=dtype)


def _genome(n, g, repeats=0.0):
    """Uniform random base codes with `repeats` of them pasted as 1 % diverged 3 kbp copies."""
    codes = _randint(0, 4, n, g, torch.uint8)
    length = 3000
    copies = int(n * repeats / length)
    if copies:  # onto places that don't overlap
        at = torch.arange(length, device="cuda")
        src, dst = _randint(0, n - length, copies, g), length * torch.randperm(n // length, generator=g, device="cuda")[:copies]
        seg = codes[src[:, None] + at]
        change = torch.rand(seg.shape, generator=g, device="cuda") < 0.01
        codes[dst[:, None] + at] = torch.where(change, (seg + 1) & 3, seg)
    return codes


def _lengths(lo, hi, n, g):
    """n read lengths spread evenly over lo..hi in random order (their sum is the same for every seed)."""
    return (lo + torch.arange(n, device="cuda") % (hi - lo + 1))[torch.randperm(n, generator=g, device="cuda")]


def _reads(codes, starts, lens, err, n_rate, g):
    """Reads of either strand from the given starts: (seq, qual, offsets); substitutions get
    Phred 2..15, right bases 25..40, N bases 2."""
    n = lens.numel()
    offs = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offs[1:])
    total = int(offs[-1])
    seq = torch.empty(total, dtype=torch.uint8, device="cuda")
    qual = torch.empty(total, dtype=torch.uint8, device="cuda")
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
    strand = _randint(0, 2, n, g).bool()
    step = max(1, 50_000_000 // max(1, int(lens.max())))
    for a in range(0, n, step):
        b = min(n, a + step)
        o0, o1 = int(offs[a]), int(offs[b])
        m, ln, rev = o1 - o0, lens[a:b], strand[a:b]
        rid = torch.repeat_interleave(torch.arange(b - a, device="cuda"), ln, output_size=m)
        at = torch.arange(m, device="cuda") - (offs[a:b] - o0)[rid]
        back = rev[rid]
        at = torch.where(back, (starts[a:b] + ln - 1)[rid] - at, starts[a:b][rid] + at)
        c = codes[at]
        c = torch.where(back, 3 - c, c)
        u = torch.rand(m, generator=g, device="cuda")
        wrong = u < err
        c = torch.where(wrong, (c + _randint(1, 4, m, g, torch.uint8)) & 3, c)
        seq[o0:o1] = letters[c.long()]
        qual[o0:o1] = 33 + torch.where(wrong, _randint(2, 16, m, g, torch.uint8), _randint(25, 41, m, g, torch.uint8))
        if n_rate > 0:
            none = u > 1.0 - n_rate
            seq[o0:o1].masked_fill_(none, ord("N"))
            qual[o0:o1].masked_fill_(none, 35)
    return seq, qual, offs


def _sample(genome, coverage, read_min, read_max, err, n_rate, repeats, satellite, g):
    """(genome codes, seq, qual, offsets) of one sample."""
    codes = _genome(genome, g, repeats)
    n = max(1, int(round(coverage * genome / (0.5 * (read_min + read_max)))))
    lens = _lengths(read_min, read_max, n, g)
    starts = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (genome - lens + 1)).long()
    if satellite:  # 30 % of the reads from a 100 kbp array of one 171 bp unit, mixed in between
        unit = _randint(0, 4, 171, g, torch.uint8)
        array = unit.repeat(585)
        ns = int(n * 3 / 7)
        ls = _lengths(read_min, read_max, ns, g)
        ss = genome + (torch.rand(ns, generator=g, device="cuda", dtype=torch.float64) * (array.numel() - ls + 1)).long()
        mix = torch.randperm(n + ns, generator=g, device="cuda")
        lens, starts = torch.cat([lens, ls])[mix], torch.cat([starts, ss])[mix]
        return (codes, *_reads(torch.cat([codes, array]), starts, lens, err, n_rate, g))
    return (codes, *_reads(codes, starts, lens, err, n_rate, g))


def _kmers(codes, at, back, changed, k, g):
    """Keys [n, 2] of the genome's k-mers at `at`, reverse-complemented where `back`, with one
    base changed where `changed`."""
    n = at.numel()
    lo, hi = torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda")
    where = torch.where(changed, _randint(0, k, n, g), torch.full((n,), -1, device="cuda"))
    shift = _randint(1, 4, n, g)
    for j in range(k):
        c = codes[torch.where(back, at + (k - 1 - j), at + j)].long()
        c = torch.where(back, 3 - c, c)
        c = torch.where(where == j, (c + shift) & 3, c)
        hi = (hi << 2) | ((lo >> 62) & 3)
        lo = (lo << 2) | c
    if k <= 32:
        hi.zero_()
    return torch.stack([lo, hi], 1).contiguous()


def _query_keys(codes, k, n, g):
    """2n keys in random order: genome k-mers of either strand, and as many with one base changed."""
    span = codes.numel() - k + 1
    at = torch.randperm(span, generator=g, device="cuda")[:n] if span <= 4 * n else _randint(0, span, n, g)
    at = at.repeat(2)
    changed = torch.arange(at.numel(), device="cuda") >= at.numel() // 2
    mix = torch.randperm(at.numel(), generator=g, device="cuda")
    return _kmers(codes, at[mix], _randint(0, 2, at.numel(), g).bool(), changed[mix], k, g)


def _params(genome, coverage, length, n_bases, n_reads, err, k, min_depth=2, bloom=True, canonical=True, satellite=False):
    """Handle parameters of a user who knows the approximate genome size, coverage and error rate."""
    windows = max(1.0, n_bases - n_reads * (k - 1.0)) if length >= k else float(n_bases)
    p_err = 1.0 - (1.0 - err) ** k
    strands = 1 if canonical else 2
    distinct = strands * genome + windows * p_err
    f = coverage * max(0.05, 1.0 - (k - 1) / length)
    lam = f * (err / 3.0) * (1.0 - err) ** (k - 1)
    twice = strands * genome * k * 3 * (1.0 - math.exp(-lam) * (1.0 + lam))
    keys = strands * genome + twice + 0.01 * windows * p_err if bloom else distinct
    if satellite:
        keys += min(0.05 * windows, 171 * k * k * 4.5 * strands) + 171 * k * 3 * strands
    return make_params(k=k, max_bases=n_bases, max_reads=n_reads, min_depth=min_depth, use_bloom=bloom, canonical=canonical,
                       expected_distinct=int(distinct * 1.05) + 1024, expected_keys=int(keys * 1.25) + 1024,
                       heavy_hitters=satellite)


def _handle(c, seq, offs, length):
    return KmerAnalysis(_params(c["genome"], c["coverage"] * (10 / 7 if c.get("satellite") else 1), length, int(seq.numel()),
                                int(offs.numel()) - 1, c["err"], c["k"], c.get("min_depth", 2), c.get("bloom", True),
                                c.get("canonical", True), c.get("satellite", False)))


def _fastq_text(seq, qual, lens, offs, crlf):
    """Four-line records with 14-character names."""
    nl = 2 if crlf else 1
    n, total = lens.numel(), seq.numel()
    start = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(2 * lens + 15 + 4 * nl, 0, out=start[1:])
    size = int(start[-1])
    text = torch.full((size,), 10, dtype=torch.uint8, device="cuda")
    at, ids = start[:-1], torch.arange(n, device="cuda")
    for j, ch in enumerate(b"@read"):
        text[at + j] = ch
    for j in range(9):
        text[at + 5 + j] = (48 + (ids // 10 ** (8 - j)) % 10).to(torch.uint8)
    plus = at + 14 + nl + lens + nl
    text[plus] = ord("+")
    if crlf:
        for e in (at + 14, at + 14 + nl + lens, plus + 1, start[1:] - nl):
            text[e] = 13
    for a in range(0, n, 500_000):
        b = min(n, a + 500_000)
        o0, o1 = int(offs[a]), int(offs[b])
        rid = torch.repeat_interleave(torch.arange(b - a, device="cuda"), lens[a:b], output_size=o1 - o0)
        pos = torch.arange(o0, o1, device="cuda") - offs[a:b][rid]
        text[(at[a:b] + 14 + nl)[rid] + pos] = seq[o0:o1]
        text[(plus[a:b] + 1 + nl)[rid] + pos] = qual[o0:o1]
    assert total == int(offs[-1])
    return text


# ------------------------------------------------------------------ cases

def _batch_specs(c):
    """Genome, coverage, read length and error rate of each sample: a fixed spread of the case's
    ranges, uneven like a sequencing run's samples."""
    n, lo, hi = c["samples"], math.log(c["genome_min"]), math.log(c["genome_max"])
    return [(int(math.exp(lo + (hi - lo) * ((0.618034 * (i + 1)) % 1.0))), 20 + 40 * ((0.754878 * (i + 1)) % 1.0),
             100 + int(151 * ((0.569840 * (i + 1)) % 1.0)), 0.005 + 0.01 * ((0.324718 * (i + 1)) % 1.0)) for i in range(n)]


def prepare(case, seed):
    c, g = case, _gen(seed, 17)
    kind = c["kind"]
    if kind == "batch":
        handles, reads, keys = [], [], []
        for genome, cov, length, err in _batch_specs(c):
            codes, seq, qual, offs = _sample(genome, cov, length, length, err, 0.0, 0.0, False, g)
            handles.append(KmerAnalysis(_params(genome, cov, length, int(seq.numel()), int(offs.numel()) - 1, err, c["k"])))
            reads.append((seq, qual, offs))
            keys.append(_query_keys(codes, c["k"], 20_000, g))
        torch.cuda.synchronize()
        return dict(kind=kind, graph=BatchGraph(handles, reads), keys=keys)
    if kind == "fastq":
        n = max(1, int(c["bases"] / (0.5 * (c["read_min"] + c["read_max"]))))
        lens = _lengths(c["read_min"], c["read_max"], n, g)
        codes = _genome(1_000_000, g)
        seq, qual, offs = _reads(codes, _randint(0, 1_000_000 - 500, n, g), lens, 0.01, 1e-4, g)
        text = _fastq_text(seq, qual, lens, offs, c["crlf"])
        return dict(kind=kind, text=text.cpu().numpy() if c["host"] else text)
    if kind == "query":
        codes, seq, qual, offs = _sample(c["genome"], 20.0, 150, 150, 0.005, 0.0, 0.0, False, g)
        ka = _handle(dict(c, coverage=20.0, err=0.005), seq, offs, 150)
        ka.count(seq, qual, offs)
        ka.finalize()
        keys = _query_keys(codes, c["k"], (c["queries"] + 1) // 2, g)[:c["queries"]].contiguous()
        return dict(kind=kind, ka=ka, keys=keys)
    codes, seq, qual, offs = _sample(c["genome"], c["coverage"], c["read_min"], c["read_max"], c["err"], c.get("n_rate", 0.0),
                                     c.get("repeats", 0.0), c.get("satellite", False), g)
    length = 0.5 * (c["read_min"] + c["read_max"])
    if kind == "estimate":
        return dict(kind=kind, k=c["k"], reads=(seq, qual, offs))
    ka = _handle(c, seq, offs, length)
    if kind == "contigs":
        ka.count(seq, qual, offs)
        ka.finalize()
        return dict(kind=kind, ka=ka, seq=np.zeros(4 * c["genome"], np.uint8), lengths=np.zeros(c["genome"] // 16, np.int64))
    state = dict(kind=kind, ka=ka, reads=(seq, qual, offs), records=c["records"], k=c["k"], host=c["host"])
    if c["records"]:  # room for the ordered records, zero behind them
        state["out"] = [torch.zeros((int(seq.numel()), *w), dtype=t, device="cuda") for w, t in
                        (((2,), torch.int64), ((), torch.int32), ((8,), torch.int32), ((2,), torch.uint8))]
    else:
        state["keys"] = _query_keys(codes, c["k"], min(MAX_QUERIES, c["genome"]), g)
    if c["host"]:
        pinned = [x.cpu().pin_memory().numpy() for x in state["reads"]]
        state["reads"] = (pinned[0], pinned[1], pinned[2].view(np.uint64))
        state["keys"] = state["keys"].cpu().pin_memory().numpy().view(np.uint64)
        rows = int(2.2 * c["genome"]) * (1 if c["canonical"] else 2) + 100_000
        state["out"] = host_result_buffers(rows if c["min_depth"] > 1 else int(seq.numel()), pinned=True)
    return state


def _answers(info, got):
    return {"n": int(info.n), "n_uu": int(info.n_uu), "windows": int(info.valid_windows), "counts": got[0], "ext": got[1], "codes": got[2]}


def run(state):
    kind = state["kind"]
    if kind == "count":
        ka = state["ka"]
        ka.reset()
        ka.count(*state["reads"])
        if state["host"]:
            ka.finalize_to_host(state["out"])
            counts, ext, codes = ka.query(state["keys"])
            return _answers(ka.result_info, (counts.view(np.int32), ext.view(np.int32), codes))
        info = ka.finalize()
        if not state["records"]:
            return _answers(info, ka.query(state["keys"]))
        keys, counts, ext, codes = ka.copy_result_device()
        if state["k"] > 31:  # order by the low word as an unsigned number, then stably by the high word
            order = torch.argsort(keys[:, 0] ^ (-1 << 63))
            order = order[torch.argsort(keys[order, 1], stable=True)]
        else:
            order = torch.argsort(keys[:, 0])
        n = len(order)
        for whole, rows in zip(state["out"], (keys, counts, ext, codes)):
            if rows.dim() == 1 or rows.shape[1] * rows.element_size() < 16:
                torch.index_select(rows, 0, order, out=whole[:n])
            else:  # 16 bytes at a time
                for to, column in zip(whole.view(torch.complex128).unbind(1), rows.view(torch.complex128).unbind(1)):
                    to[:n] = column[order]
        return {"n": int(info.n), "n_uu": int(info.n_uu), "windows": int(info.valid_windows), "records": state["out"]}
    if kind == "batch":
        graph = state["graph"]
        graph.replay()
        infos = graph.results()
        with torch.cuda.stream(graph.stream):
            answers = [h.query(q) for h, q in zip(graph.handles, state["keys"])]
        return {"n": np.array([int(i.n) for i in infos]), "n_uu": np.array([int(i.n_uu) for i in infos]),
                "windows": np.array([int(i.valid_windows) for i in infos]), "answers": [list(a) for a in answers]}
    if kind == "query":
        return list(state["ka"].query(state["keys"]))
    if kind == "estimate":
        e = estimate_distinct(*state["reads"], k=state["k"])
        return {"distinct": e.distinct, "registers": e.registers, "valid_windows": e.valid_windows, "sampled_windows": e.sampled_windows,
                "bucket_windows": e.bucket_windows.view(np.int64), "heavy": int(e.heavy_hitters)}
    if kind == "fastq":
        return list(parse_fastq(state["text"]))
    strings, info = state["ka"].contigs()
    strings.sort()  # contigs come in unspecified order
    raw = np.frombuffer("".join(strings).encode(), dtype=np.uint8)
    state["seq"][:raw.size] = raw
    state["lengths"][:len(strings)] = [len(s) for s in strings]
    return {"seq": state["seq"], "lengths": state["lengths"], "contigs": len(strings), "vertices": info["n_vertices"],
            "cycles": info["n_cycles"]}


def work(case):
    """Bytes: reads (base and quality), offsets and keys read once; records and answers written once."""
    c, kind = case, case["kind"]
    if kind == "batch":
        return {"bytes": sum(2.0 * g * cov + 8 * g * cov / ln + 54.0 * g + 40_000 * 54.0 for g, cov, ln, _ in _batch_specs(c)), "flops": 0}
    if kind == "query":
        return {"bytes": c["queries"] * (16.0 + 38.0), "flops": 0}
    length = 0.5 * (c["read_min"] + c["read_max"])
    if kind == "fastq":
        n = c["bases"] / length
        return {"bytes": n * (2 * length + 15 + (8 if c["crlf"] else 4)) + 2.0 * c["bases"] + 8 * n, "flops": 0}
    bases = c["genome"] * c["coverage"] * (10 / 7 if c.get("satellite") else 1)
    if kind == "estimate":
        return {"bytes": bases + 8 * bases / length, "flops": 0}
    if kind == "contigs":
        return {"bytes": c["genome"] * (18.0 + 1.0), "flops": 0}
    looked_up = 0 if c["records"] else 2 * min(MAX_QUERIES, c["genome"])
    return {"bytes": 2 * bases + 8 * bases / length + 54.0 * c["genome"] + 54.0 * looked_up, "flops": 0}


# ------------------------------------------------------------------ the sketch in plain torch

def _signed(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _shr(x, s):
    return (x >> s) & ((1 << (64 - s)) - 1)


def _fmix(x):
    """The 64-bit finaliser of MurmurHash3 on int64 words."""
    x = (x ^ _shr(x, 33)) * _signed(0xff51afd7ed558ccd)
    x = (x ^ _shr(x, 33)) * _signed(0xc4ceb9fe1a85ec53)
    return x ^ _shr(x, 33)


def exact(case, seed):
    """The estimate from a HyperLogLog sketch of every valid window, made with plain torch and
    summed in 64 bits. The other cases' outputs are whole numbers."""
    c = case
    if c["kind"] != "estimate" or c["genome"] * c["coverage"] > 4e8:
        return None
    k, p = c["k"], 14
    _, seq, _, offs = _sample(c["genome"], c["coverage"], c["read_min"], c["read_max"], c["err"], 0.0, 0.0, False, _gen(seed, 17))
    code = ((seq >> 1) ^ (seq >> 2)).long() & 3
    best = torch.zeros(1 << p, dtype=torch.int64, device="cuda")
    sign = -1 << 63
    for a in range(0, seq.numel() - k + 1, 20_000_000):
        n = min(20_000_000, seq.numel() - k + 1 - a)
        at = torch.arange(a, a + n, device="cuda")
        read = torch.searchsorted(offs, at, right=True)
        ok = at + k <= offs[read]
        lo, hi, rlo, rhi = (torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(4))
        for j in range(k):
            f, r = code[a + j:a + j + n], 3 - code[a + k - 1 - j:a + k - 1 - j + n]
            hi, lo = (hi << 2) | ((lo >> 62) & 3), (lo << 2) | f
            rhi, rlo = (rhi << 2) | ((rlo >> 62) & 3), (rlo << 2) | r
        keep = (hi < rhi) | ((hi == rhi) & ((lo ^ sign) <= (rlo ^ sign)))
        lo, hi = torch.where(keep, lo, rlo)[ok], torch.where(keep, hi, rhi)[ok]
        h = _fmix(lo ^ (hi * _signed(0x9e3779b97f4a7c15) + 0x632be59bd9b4e019))
        rest = (h & ((1 << (64 - p)) - 1)).double()
        rank = torch.where(rest > 0, (64 - p) - torch.frexp(rest).exponent.long() + 1, torch.full_like(h, 64 - p + 1))
        best.scatter_reduce_(0, _shr(h, 64 - p), rank, "amax")
    m = float(1 << p)
    raw = 0.7213 / (1.0 + 1.079 / m) * m * m / float(torch.exp2(-best.double()).sum())
    zeros = int((best == 0).sum())
    value = m * math.log(m / zeros) if raw <= 2.5 * m and zeros else raw
    return {"distinct": value, "registers": None, "valid_windows": None, "sampled_windows": None, "bucket_windows": None, "heavy": None}
