"""The work that users of this package have it do, as cases that can be timed.

A case is one pass through the public entry points: the whole path from reads
to the SdBG (mh_pack_reads, mh_count_kmers, mh_mercy_kmers, mh_build_sdbg), one
of its calls alone, the multiple-k iteration, a batch of read sets, or the
no-allocation sort.  Reads are made on the GPU from the seed: sampled from
random genomes with substitution errors, as the package's own generators
(``synth``) make them.

listed()  the cases; draw(rng) one more of the same ranges
prepare   the inputs of a case and what a user's program keeps beside them
run       one pass, all its outputs, in buffers of a fixed size that the program
          keeps (an output's size depends on the reads; the rest stays zero)
work      bytes the pass cannot do without (inputs read once, outputs written once)
exact     the same outputs from plain torch, where that is quick

Every output is a whole number: keys, counts, codes, bits and offsets.
"""
import math

import numpy as np
import torch

import paper_1409_7208_gb300 as mh
from paper_1409_7208_gb300 import multik

DEV = "cuda:0"

# Read sets ------------------------------------------------------------
# reads    number of reads (pairs: two reads each of 'len_hi' bases)
# len_lo, len_hi   read lengths, uniform (pairs: all of len_hi)
# genomes, genome  number of genomes and their (median) length; one genome:
#                  uniform positions; several: lengths and abundances at the
#                  quantiles of lognormals (sigma 0.5 and 1.5), as a community
#                  has, so that sets of one case differ little in size
# err      substitution rate; pairs: of the 3' end, rising from 0
# n_rate   chance of an N in place of a base


def listed():
    return [
        # The smallest job, one isolate's amplicon-sized genome at 20x: latency and launches.
        dict(name="path_small", kind="path", reads=10_000, len_lo=100, len_hi=100, pairs=False, genomes=1,
             genome=50_000, err=0.01, n_rate=0.0, k=21, d=2, host=False, mult=False),
        # The median job of a request stream: ragged reads in pinned host memory, two key words.
        dict(name="path_job_host", kind="path", reads=447_213, len_lo=100, len_hi=150, pairs=False, genomes=1,
             genome=2_000_000, err=0.01, n_rate=0.0, k=41, d=2, host=True, mult=False),
        # An ordinary metagenome set, some reads with N.
        dict(name="path_set", kind="path", reads=2_000_000, len_lo=150, len_hi=150, pairs=True, genomes=10,
             genome=2_000_000, err=0.01, n_rate=0.0005, k=31, d=2, host=False, mult=False),
        # The largest: a whole metagenome of 3 Gbp in one pass.
        dict(name="path_metagenome", kind="path", reads=20_000_000, len_lo=150, len_hi=150, pairs=True,
             genomes=100, genome=2_000_000, err=0.01, n_rate=0.0, k=31, d=2, host=False, mult=False),
        # Counting alone at a middle k (two key words) and at a large one (four).
        dict(name="count_k61", kind="count", reads=3_000_000, len_lo=100, len_hi=150, pairs=False, genomes=1,
             genome=15_000_000, err=0.01, n_rate=0.0, k=61, d=2, host=False, mult=False),
        dict(name="count_k99", kind="count", reads=4_000_000, len_lo=150, len_hi=150, pairs=True, genomes=10,
             genome=2_000_000, err=0.01, n_rate=0.0, k=99, d=2, host=False, mult=False),
        # Mercy edges of a low-coverage community, where they matter most.
        dict(name="mercy_k31", kind="mercy", reads=3_000_000, len_lo=150, len_hi=150, pairs=True, genomes=20,
             genome=2_000_000, err=0.01, n_rate=0.0, k=31, d=2, host=False, mult=False),
        # The graph with edge multiplicities, as cleaning wants them.
        dict(name="build_k47_mult", kind="build", reads=3_000_000, len_lo=150, len_hi=150, pairs=True, genomes=10,
             genome=2_000_000, err=0.01, n_rate=0.0, k=47, d=2, host=False, mult=True),
        # Packing of reads as they come off a sequencer: ragged after trimming, with Ns.
        dict(name="pack_ragged_n", kind="pack", reads=5_000_001, len_lo=30, len_hi=151, pairs=False, genomes=1,
             genome=5_000_000, err=0.01, n_rate=0.002, k=31, d=2, host=False, mult=False),
        # The multiple-k iteration: every key width, contigs carried from k to k.
        dict(name="iterate", kind="iterate", reads=2_000_000, len_lo=100, len_hi=100, pairs=False, genomes=1,
             genome=10_000_000, err=0.01, n_rate=0.0, ks="27,47,67,87,99", d=2, walks=16_384, max_len=10_000,
             host=False, mult=False),
        # Independent sets at once on worker streams, sizes as a batch has them.
        dict(name="batch", kind="batch", sets=6, reads=300_000, len_lo=150, len_hi=150, pairs=True, genomes=10,
             genome=2_000_000, err=0.01, n_rate=0.0, k=31, d=2, workers=4, host=False, mult=False),
        # The sort offered to callers that may not allocate.
        dict(name="sort_noalloc", kind="sort", n=300_007, nw=1, bits=62),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "path", "path", "count", "count", "mercy", "build", "pack", "iterate", "batch", "sort"])
    if kind == "sort":
        nw = rng.choice([1, 2, 4])
        return dict(kind="sort", n=_log_int(rng, 500, (1 << 21) // nw), nw=nw,
                    bits=2 * (rng.randint(20 if nw == 1 else 16 * nw + 1, 32 * nw)))
    k = rng.choice([rng.randint(15, 31), 21, 27, 31, rng.randint(32, 63), 41, 47, 61, rng.randint(64, 99), 67, 87])
    nw = 1 if k <= 31 else 2 if k <= 63 else 4
    most = {"path": 12e6, "count": 12e6, "mercy": 8e6, "build": 8e6, "pack": 12e6, "iterate": 2e6, "batch": 3e5}[kind]
    least = {"path": 1e4, "count": 1e4, "mercy": 1e5, "build": 1e5, "pack": 1e4, "iterate": 5e4, "batch": 2e4}[kind]
    pairs = rng.random() < 0.5
    reads = _log_int(rng, least, most / (nw if kind != "iterate" else 1))
    c = dict(kind=kind, reads=reads // 2 * 2 if pairs else reads, pairs=pairs, d=rng.choice([2, 2, 2, 3]),
             n_rate=rng.choice([0.0, 0.0, 0.001]), err=rng.choice([0.005, 0.01]), host=False, mult=False)
    if pairs:
        c["len_lo"] = c["len_hi"] = rng.choice([100, 125, 150])
        c["genomes"] = rng.choice([5, 10, 20, 50])
        c["genome"] = rng.randint(500_000, 2_000_000)
    else:
        c["len_hi"] = rng.randint(100, 151)
        c["len_lo"] = rng.choice([c["len_hi"], rng.randint(50, c["len_hi"])])
        c["genomes"] = 1
        c["genome"] = max(20_000, c["reads"] * c["len_hi"] // rng.randint(5, 40))
    if kind == "iterate":
        c.update(ks=rng.choice(["21,41,61", "27,47,67,87", "31,51,71,91"]), d=2, walks=_log_int(rng, 500, 16_384),
                 max_len=rng.randint(1_000, 10_000))
        return c
    c["k"] = k
    if kind == "path":
        c["host"] = rng.random() < 0.3
    if kind == "build":
        c["mult"] = rng.random() < 0.5
    if kind == "batch":
        c.update(sets=rng.randint(2, 6), workers=rng.randint(1, 6))
    return c


# Inputs -----------------------------------------------------------------

def _community(case):
    """Lengths of the genomes and the share of the reads each gets."""
    G = case["genomes"]
    if G == 1:
        return np.array([max(case["genome"], 2000)]), np.ones(1)
    z = torch.special.ndtri((torch.arange(G, dtype=torch.float64) + 0.5) / G).numpy()
    lens = np.maximum(2000, case["genome"] * np.exp(0.5 * z)).astype(np.int64)
    weight = lens * np.exp(1.5 * z[np.random.RandomState(7).permutation(G)])
    return lens, weight / weight.sum()


def _sample(case, reads, seed):
    """(ascii uint8, offs int64) on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    L, G = case["len_hi"], case["genomes"]
    lens, share = _community(case)
    lens, cdf = torch.from_numpy(lens).to(DEV), torch.from_numpy(np.cumsum(share)).to(DEV)
    first = torch.cumsum(lens, 0) - lens
    codes = torch.randint(0, 4, (int(lens.sum()),), generator=g, device=DEV, dtype=torch.uint8)
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)
    at = torch.arange(L, device=DEV, dtype=torch.int32)
    ramp = (at + 0.5) / L if case["pairs"] else torch.ones(L, device=DEV)
    out, out_len = [], []
    for c0 in range(0, reads, 1_000_000):
        n = min(1_000_000, reads - c0)
        units = n // 2 if case["pairs"] else n
        which = torch.searchsorted(cdf, rand(units).double()).clamp_(max=G - 1)
        room = lens[which]
        if case["pairs"]:
            size = (350 + 35 * torch.randn(units, generator=g, device=DEV)).round().long().clamp_(L, 1500)
        else:
            size = torch.full((units,), L, device=DEV)
        start = (first[which] + (rand(units).double() * (room - size + 1)).long()).int()
        flip = rand(units) < 0.5
        if case["pairs"]:
            # mate 1 from the fragment's front, mate 2 the reverse complement of its end; either strand first
            start = torch.stack([start, start + (size - L).int()], 1)
            back = torch.stack([torch.zeros_like(flip), torch.ones_like(flip)], 1)
            start = torch.where(flip[:, None], start.flip(1), start).reshape(-1)
            flip = torch.where(flip[:, None], back.flip(1), back).reshape(-1)
        pos = start[:, None] + torch.where(flip[:, None], L - 1 - at, at)
        b = codes.index_select(0, pos.reshape(-1)).reshape(n, L)
        del pos
        b = torch.where(flip[:, None], 3 - b, b)
        hit = rand(n, L) < case["err"] * ramp
        b = torch.where(hit, (b + torch.randint(1, 4, (n, L), generator=g, device=DEV, dtype=torch.uint8)) & 3, b)
        del hit
        a = letters.index_select(0, b.reshape(-1).int()).reshape(n, L)
        if case["n_rate"]:
            a = torch.where(rand(n, L) < case["n_rate"], torch.full_like(a, ord("N")), a)
        if case["len_lo"] < L:
            ln = torch.randint(case["len_lo"], L + 1, (n,), generator=g, device=DEV)
            a = a[at < ln[:, None]]
        else:
            ln = torch.full((n,), L, device=DEV)
        out.append(a.reshape(-1))
        out_len.append(ln)
    offs = torch.zeros(reads + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.cat(out_len), 0, out=offs[1:])
    return torch.cat(out), offs


# Sizes ----------------------------------------------------------------------

def _nw(k):
    return 1 if k <= 31 else 2 if k <= 63 else 4


def _shape(case, reads):
    """Reads and bases of a set."""
    return reads, reads * (case["len_lo"] + case["len_hi"]) / 2


def _at_least(lam, d):
    """Chance that a Poisson count is at least d."""
    return 1 - sum(math.exp(-lam) * lam ** i / math.factorial(i) for i in range(d)) if lam < 500 else 1.0


def _solid(case, reads, k):
    """Expected solid (k+1)-mers of a set, both strands: those of the genomes
    seen at least d times without an error, and those with one error made at
    least d times alike."""
    reads, bases = _shape(case, reads)
    windows = max(0.0, bases - reads * k)
    err = case["err"] * (0.5 if case["pairs"] else 1.0)
    total = 0.0
    for size, share in zip(*_community(case)):
        c = windows * share / size
        total += size * (_at_least(c * (1 - err) ** (k + 1), case["d"])
                         + 3 * (k + 1) * _at_least(c * err / 3 * (1 - err) ** k, case["d"]))
    return 2 * total, windows


def _room(case, reads, k):
    """Buffers' entries for (solid, mercy, dummy entries): well above what the sets of a case give."""
    solid, windows = _solid(case, reads, k)
    walked = case["walks"] * case["max_len"] // 4 if case["kind"] == "iterate" else 0
    s = int(min(1.3 * solid + walked, windows + 8 * walked)) + 50_000
    return s, int(0.3 * min(s, windows)) + 50_000, int(0.3 * s) + 50_000


def _kmer_buffers(n, k):
    return [torch.zeros(n * _nw(k), dtype=torch.int64, device=DEV), torch.zeros(n, dtype=torch.int32, device=DEV)]


def _graph_buffers(case, s, m, t, k):
    E = s + m + 2 * t
    words = (E + 31) // 32
    b = [torch.zeros(E, dtype=torch.uint8, device=DEV)]
    b += [torch.zeros(words, dtype=torch.int32, device=DEV) for _ in range(3)]
    b += [torch.zeros(t * _nw(k), dtype=torch.int64, device=DEV)]
    return b + ([torch.zeros(E, dtype=torch.int32, device=DEV)] if case["mult"] else [])


def _contig_buffers(case):
    return [torch.zeros(case["walks"] * case["max_len"], dtype=torch.uint8, device=DEV),
            torch.zeros(case["walks"] + 1, dtype=torch.int64, device=DEV)]


def _buffers(case, reads):
    kind = case["kind"]
    if kind == "pack":
        n, bases = _shape(case, reads)
        # an N ends a fragment; the last one starts no other
        return [torch.zeros(int(1.02 * bases / 16) + 1000, dtype=torch.int32, device=DEV),
                torch.zeros(int(n + 1.1 * bases * case["n_rate"]) + 1000, dtype=torch.int64, device=DEV),
                torch.zeros(int(n + 1.1 * bases * case["n_rate"]) + 1000, dtype=torch.int32, device=DEV)]
    out = []
    for k in [int(x) for x in case["ks"].split(",")] if kind == "iterate" else [case["k"]]:
        s, m, t = _room(case, reads, k)
        if kind != "build":
            out += _kmer_buffers(m if kind == "mercy" else s, k)
        if kind in ("path", "batch", "iterate"):
            out += _kmer_buffers(m, k)
        if kind in ("path", "batch", "iterate", "build"):
            out += _graph_buffers(case, s, m, t, k)
        if kind == "iterate":
            out += _contig_buffers(case)
    return out


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 16 * case["n"] * case["nw"], "flops": 0}
    reads, bases = _shape(case, case["reads"])
    ascii, packed = bases + 8 * reads, bases / 4 + 8 * reads
    if kind == "pack":
        return {"bytes": int(ascii + packed + 4 * reads), "flops": 0}
    total = 0.0
    for k in [int(x) for x in case["ks"].split(",")] if kind == "iterate" else [case["k"]]:
        S = min(_solid(case, case["reads"], k))
        table, graph = S * (8 * _nw(k) + 4), S * (1.375 + (4 if case["mult"] else 0))
        total += {"path": ascii + table + graph, "batch": ascii + table + graph, "iterate": ascii + table + graph,
                  "count": packed + table, "mercy": packed + table, "build": table + graph}[kind]
    if kind == "iterate":
        total += len(case["ks"].split(",")) * case["walks"] * case["max_len"]
    return {"bytes": int(total * case.get("sets", 1)), "flops": 0}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        g = torch.Generator(device=DEV).manual_seed(seed)
        nw, bits = case["nw"], case["bits"]
        keys = torch.randint(-(1 << 63), (1 << 63) - 1, (case["n"], nw), generator=g, device=DEV, dtype=torch.int64)
        for w in range(nw):  # the low `bits` bits of a key are in use
            left = min(64, max(0, bits - 64 * w))
            if left < 64:
                keys[:, w] &= (1 << left) - 1
        return dict(case=case, keys=keys.reshape(-1), out=torch.empty(case["n"] * nw, dtype=torch.int64, device=DEV))
    s = dict(case=case, ctx=mh.Context(device=0, with_mult=case["mult"]))
    if kind == "batch":
        # sizes spread about the case's number of reads, a factor of four either way
        rng = np.random.default_rng(seed)
        n = (case["reads"] * np.exp(rng.uniform(-1.386, 1.386, case["sets"]))).astype(int) // 2 * 2
        s["sets"] = [_sample(case, int(x), seed * 1000 + i) for i, x in enumerate(n)]
        s["out"] = [b for _ in n for b in _buffers(case, 4 * case["reads"])]
        return s
    ascii, offs = _sample(case, case["reads"], seed)
    if case["host"]:
        ascii, offs = ascii.cpu().pin_memory(), offs.cpu().pin_memory()
    s.update(ascii=ascii, offs=offs, out=_buffers(case, case["reads"]))
    if kind in ("count", "mercy", "build"):
        s["reads"] = mh.mh_pack_reads(s["ctx"], ascii, offs)
    if kind in ("mercy", "build"):
        s["solid"] = mh.mh_count_kmers(s["ctx"], s["reads"], case["k"], case["d"])
    if kind == "build":
        s["mercy"] = mh.mh_mercy_kmers(s["ctx"], s["reads"], s["solid"])
    return s


# One pass -----------------------------------------------------------------

def _kmers(h):
    return [h.keys, h.counts]


def _graph(h):
    t = h.tensors()
    out = [t[f] for f in ("W", "last", "valid", "dummy", "aux")]
    return (out if t["mult"] is None else out + [t["mult"]]), t["F"]


def _keep(state, got, numbers):
    """The outputs into the program's own buffers; their sizes and the other numbers as one array."""
    for b, x in zip(state["out"], got, strict=True):
        if x.numel() > b.numel():
            raise ValueError("an output of %d entries, a buffer of %d" % (x.numel(), b.numel()))
        b[:x.numel()].copy_(x.reshape(-1))
    return state["out"] + [np.array([x.numel() for x in got] + numbers, dtype=np.int64)]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sort":
        mh.mh_sort_keys_noalloc(state["keys"], state["out"], case["nw"], case["bits"])
        return state["out"]
    ctx = state["ctx"]
    if kind == "path":
        reads = mh.mh_pack_reads(ctx, state["ascii"], state["offs"])
        solid = mh.mh_count_kmers(ctx, reads, case["k"], case["d"])
        mercy = mh.mh_mercy_kmers(ctx, reads, solid)
        graph, F = _graph(mh.mh_build_sdbg(ctx, solid, mercy))
        return _keep(state, _kmers(solid) + _kmers(mercy) + graph, F)
    if kind == "count":
        solid = mh.mh_count_kmers(ctx, state["reads"], case["k"], case["d"])
        v = solid.view()
        return _keep(state, _kmers(solid), [v.n_kmers, v.n_distinct])
    if kind == "mercy":
        return _keep(state, _kmers(mh.mh_mercy_kmers(ctx, state["reads"], state["solid"])), [])
    if kind == "build":
        return _keep(state, *_graph(mh.mh_build_sdbg(ctx, state["solid"], state["mercy"])))
    if kind == "pack":
        t = mh.mh_pack_reads(ctx, state["ascii"], state["offs"]).tensors()
        return _keep(state, [t["packed"], t["frag_offs"], t["frag_read"]], [t["n_packed"]])
    got, numbers = [], []
    if kind == "iterate":
        for st in multik.iterate(ctx, state["ascii"], state["offs"], [int(x) for x in case["ks"].split(",")],
                                 case["d"], case["walks"], case["max_len"], seed=3, keep=True):
            t = st["contigs"].tensors()
            graph, F = _graph(st["sdbg"])
            got += _kmers(st["solid"]) + _kmers(st["mercy"]) + graph + [t["ascii"], t["offs"]]
            numbers += F
    else:
        for r in mh.mh_run_batch(ctx, state["sets"], case["k"], case["d"], workers=case["workers"]):
            graph, F = _graph(r["sdbg"])
            got += _kmers(r["solid"]) + _kmers(r["mercy"]) + graph
            numbers += F
    return _keep(state, got, numbers)


def exact(case, seed):
    """Plain torch, where that is quick: the sort by stable sorts from the
    lowest word up, a count by sorting every window's key (one-word keys)."""
    if case["kind"] == "sort":
        keys = prepare(case, seed)["keys"].reshape(case["n"], case["nw"])
        for w in range(case["nw"]):  # the sign bit flipped: unsigned order
            keys = keys[torch.argsort(keys[:, w] ^ -(1 << 63), stable=True)]
        return keys.reshape(-1)
    if case["kind"] == "count" and case["k"] <= 30 and case["reads"] <= 1_000_000:
        K, (ascii, offs) = case["k"] + 1, _sample(case, case["reads"], seed)
        code = torch.full((256,), 4, dtype=torch.int64, device=DEV)
        code[list(b"ACGT")] = torch.arange(4, device=DEV)
        base = code[ascii.int()]
        n = base.numel() - K + 1
        read = torch.repeat_interleave(torch.arange(offs.numel() - 1, device=DEV), offs.diff())
        ok = read[:n] == read[K - 1:]
        fwd, rev = torch.zeros(n, dtype=torch.int64, device=DEV), torch.zeros(n, dtype=torch.int64, device=DEV)
        for i in range(K):
            b = base[i:i + n]
            ok &= b < 4
            fwd = fwd * 4 + (b & 3)
            rev += (3 - (b & 3)) << (2 * i)
        keys, counts = torch.unique(torch.cat([fwd[ok], rev[ok]]), return_counts=True)
        keep = counts >= case["d"]
        got = [keys[keep], counts[keep].int()]
        out = _buffers(case, case["reads"])
        for b, x in zip(out, got):
            b[:x.numel()] = x
        return out + [np.array([x.numel() for x in got] + [2 * int(ok.sum()), int(keys.numel())], dtype=np.int64)]
    return None
