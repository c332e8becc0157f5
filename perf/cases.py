"""The work users have this library do, as cases to time: batched exact matching
(search, search + locate, search then locate, from device and from host
buffers) over small and large, iid, repetitive and human-like references, and
the building of an index.  Sizes and shapes follow the workloads of
datagen.py, bench.py and serve.py.

A case is a dict of plain values:

  kind      search   sa_search_batch on device buffers (counts only)
            locate   sa_search_locate on device buffers, outputs allocated once
            twocall  sa_search_batch, then sa_locate into arrays allocated once
            host     sa_search_locate from pinned host buffers into pinned ones
            build    sa_build of a text on the device, then its suffix array
  n, refs   bases of all references together, and their number (several
            references are sized 5 : 12 : 25 : 50)
  width     suffix-array width in bits
  text      iid, dup (segmental duplications and tandem repeats) or human (GC
            0.41, repeat families, tandem repeats)
  nq, m0, m1  queries of m0 .. m1 bases, drawn uniformly
  sampled   share of the queries copied from their reference (the rest random)
  subs      substitutions in a copied query: 0 .. subs
  with_n    share of the queries that hold an N, as reads do (invalid here)
  cap       positions located per query at most
  strand    each query names its strand (reads come from both)
  q_range   the caller states the batch's base range, as serve.py does

References of more than 2^28 bases are drawn once and their index is kept, as
a program keeps its genome's index resident: three such indexes would not fit
the card.  Everything else is drawn from the seed."""
import gc
import math

import torch

from paper_1303_3692_gb300 import sa

_DEV = "cuda"
_SLOT = 6000      # a repeat family's long unit
_SUB = 300        # its short unit
_SHARES = (5, 12, 25, 50)
_KEEP_ABOVE = 1 << 28
_GENOME_SEED = 1303369200

_FIELDS = dict(kind="search", n=1_000_000, refs=1, width=32, text="iid", nq=0, m0=0, m1=0, sampled=0.8, subs=0,
               with_n=0.0, cap=0, strand=False, q_range=False)


def _case(name, **kw):
    c = dict(_FIELDS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest request a server sees: a handful of reads, one bacterial
        # genome, where the call's latency is all there is
        _case("request-20", n=5_000_000, nq=20, m0=20, m1=300, sampled=0.75),
        # the paper's plain method at its smallest: 1 Mbp, 10^5 queries of 32
        _case("plain-1m", n=1_000_000, nq=100_000, m0=32, m1=32, sampled=0.5),
        # a coalesced batch of a serving process: four resident genomes, both
        # strands, ragged lengths, up to 16 positions each
        _case("serving-20k", kind="locate", n=92_000_000, refs=4, text="dup", nq=20_011, m0=20, m1=300, sampled=0.75,
              subs=1, cap=16, strand=True, q_range=True),
        # seeds and primers looked up by a mapper: shorter and longer than the
        # index's k, many positions each, with the two-call interface
        _case("seeds-100m", kind="twocall", n=100_000_003, text="human", nq=2_000_003, m0=8, m1=31, sampled=1.0,
              cap=32),
        # sequencing reads against a repetitive 100 Mbp genome; a few hold an N
        _case("reads-100m", kind="locate", n=100_000_000, text="dup", nq=10_000_000, m0=100, m1=100, subs=2,
              with_n=0.002, cap=64),
        # several genomes in one call, lengths 20 to 250 (metagenomics), counts
        _case("multi-genome", n=92_000_000, refs=4, text="dup", nq=16_000_000, m0=20, m1=250, sampled=0.7),
        # the paper's own shape: 10^7 bases, 1024-base queries, counts
        _case("paper-1024", n=10_000_000, text="human", nq=1 << 20, m0=1024, m1=1024, sampled=0.5),
        # a plant-sized genome, whose index is past the address-translation
        # reach, with paired reads of either strand
        _case("genome-430m", kind="locate", n=430_000_000, text="human", nq=9_000_001, m0=100, m1=151, sampled=0.9,
              subs=1, cap=8, strand=True, with_n=0.001),
        # the headline: a human-sized genome, 64-bit suffix array, 150-base reads
        _case("human-3.1g", kind="locate", n=3_100_000_000, width=64, text="human", nq=40_000_000, m0=150, m1=150,
              sampled=0.909, subs=1, cap=16),
        # the same kind of work from a program that holds its reads on the host
        _case("host-reads", kind="host", n=100_000_000, text="dup", nq=3_000_001, m0=100, m1=100, subs=2,
              with_n=0.002, cap=16),
        # indexing a genome, ordinary and large
        _case("build-100m", kind="build", n=100_000_000, text="human"),
        _case("build-600m", kind="build", n=600_000_011, text="human", width=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "locate", "locate", "locate", "twocall", "host", "build"])
    width = rng.choice([32, 32, 64])
    text = rng.choice(["iid", "dup", "human", "human"])
    if kind == "build":
        return _case(None, kind=kind, n=_log(rng, 1_000_000, 500_000_000) | 1, width=width, text=text)
    big = rng.random() < 0.2  # the resident human-sized genome
    refs = 1 if big else rng.choice([1, 1, 1, 4])
    n = 3_100_000_000 if big else _log(rng, 1_000_000, 250_000_000)
    m0 = _log(rng, 8, 300)
    m1 = m0 if rng.random() < 0.4 else min(1024, m0 + _log(rng, 1, 300))
    strand = rng.random() < 0.25
    most = 2_000_000_000 // (m0 + m1)  # at most 10^9 bases a batch
    most = min(most, 4_000_000 if kind == "host" else 8_000_000)
    return _case(None, kind=kind, n=n, refs=refs, width=64 if big else width, text="human" if big else text,
                 nq=_log(rng, 1, most), m0=m0, m1=m1, sampled=round(rng.uniform(0.5, 1.0), 3), subs=rng.choice([0, 1, 2]),
                 with_n=rng.choice([0.0, 0.0, 0.002]), cap=0 if kind == "search" else rng.choice([1, 8, 16, 64]),
                 strand=strand, q_range=rng.random() < 0.5 and kind != "host")


def _ref_sizes(case):
    n, k = case["n"], case["refs"]
    if k == 1:
        return [n]
    w = [_SHARES[i % len(_SHARES)] for i in range(k)]
    s = [max(2000, n * x // sum(w)) for x in w]
    return s


def _rand(g, *shape):
    return torch.rand(*shape, device=_DEV, generator=g)


def _ints(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, device=_DEV, dtype=torch.uint8, generator=g)


def _mutated(g, block, rate):
    return torch.where(_rand(g, *block.shape) < rate, (block + _ints(g, 1, 4, *block.shape)) & 3, block)


def _codes(g, n, text):
    """Codes 0..3 of one reference, drawn slot by slot (no slot overlaps
    another, so the text depends on the seed alone)."""
    gc_ = 0.41 if text == "human" else 0.5
    cons_long, cons_short = _ints(g, 0, 4, 4, _SLOT), _ints(g, 0, 4, 4, _SUB)
    n_slots = -(-n // _SLOT)
    out = torch.empty(n_slots * _SLOT, dtype=torch.uint8, device=_DEV)
    for a in range(0, n_slots, 1 << 13):
        k = min(n_slots - a, 1 << 13)
        u = _rand(g, k, _SLOT)
        c = (u >= (1 - gc_) / 2).to(torch.uint8)
        c += u >= 0.5
        c += u >= (1 + gc_) / 2
        del u
        sub = c.view(k * (_SLOT // _SUB), _SUB)
        if text == "human":  # 45 % repeat families, 10-20 % apart, half from each unit size
            pick = torch.nonzero(_rand(g, sub.shape[0]) < 0.29)[:, 0]
            fam = torch.randint(0, 4, (pick.numel(),), device=_DEV, generator=g)
            sub[pick] = _mutated(g, cons_short[fam], _rand(g, pick.numel(), 1) * 0.1 + 0.1)
        if text in ("human", "dup"):  # tandem repeats of units of 2-6 bases
            pick = torch.nonzero(_rand(g, sub.shape[0]) < (0.03 if text == "human" else 0.02))[:, 0]
            unit = torch.randint(2, 7, (pick.numel(), 1), device=_DEV, generator=g)
            at = torch.arange(_SUB, device=_DEV)[None, :] % unit
            sub[pick] = torch.gather(_ints(g, 0, 4, pick.numel(), 6), 1, at)
        if text == "human":
            pick = torch.nonzero(_rand(g, k) < 0.225)[:, 0]
            fam = torch.randint(0, 4, (pick.numel(),), device=_DEV, generator=g)
            c[pick] = _mutated(g, cons_long[fam], _rand(g, pick.numel(), 1) * 0.1 + 0.1)
        if text == "dup":  # 10 % segmental duplications, 1 % apart
            pick = torch.nonzero(_rand(g, k) < 0.10)[:, 0]
            src = torch.randint(0, k, (pick.numel(),), device=_DEV, generator=g)
            c[pick] = _mutated(g, c[src], 0.01)
        out[a * _SLOT:(a + k) * _SLOT] = c.view(-1)
    return out[:n]


def _ascii(codes):
    return torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device=_DEV)[codes.to(torch.int32)]


def _to_ascii(codes):
    out = torch.empty_like(codes)
    for a in range(0, codes.numel(), 1 << 27):
        out[a:a + (1 << 27)] = _ascii(codes[a:a + (1 << 27)])
    return out


class _Genomes:
    """The references of a case: their codes, one after the other, and an index of each."""

    def __init__(self, case, seed):
        g = torch.Generator(device=_DEV).manual_seed(seed)
        self.sizes = _ref_sizes(case)
        parts = [_codes(g, n, case["text"]) for n in self.sizes]
        self.codes = parts[0] if len(parts) == 1 else torch.cat(parts)
        self.indexes = []
        for p in parts:
            text = _to_ascii(p)
            torch.cuda.empty_cache()  # the library allocates outside torch's cache
            self.indexes.append(sa.sa_build(text, width=case["width"]))
            del text
        torch.cuda.empty_cache()


_resident = {}  # at most one: the index of a program's genome


def _genomes(case, seed):
    if case["n"] <= _KEEP_ABOVE:
        if _resident:
            _resident.clear()
            gc.collect()
        return _Genomes(case, seed)
    key = (case["n"], case["refs"], case["width"], case["text"])
    if key not in _resident:
        _resident.clear()
        gc.collect()
        torch.cuda.empty_cache()
        _resident[key] = _Genomes(case, _GENOME_SEED)
    return _resident[key]


def _queries(case, genomes, g):
    """(bases, offsets, q_ref or None) of the batch, on the GPU."""
    nq, m0, m1 = case["nq"], case["m0"], case["m1"]
    m = torch.randint(m0, m1 + 1, (nq,), device=_DEV, generator=g)
    offsets = torch.zeros(nq + 1, dtype=torch.int64, device=_DEV)
    torch.cumsum(m, 0, out=offsets[1:])
    ref = torch.randint(0, case["refs"], (nq,), device=_DEV, generator=g)
    other = (_rand(g, nq) < 0.5) if case["strand"] else torch.zeros(nq, dtype=torch.bool, device=_DEV)
    sizes = torch.tensor(genomes.sizes, device=_DEV)
    firsts = torch.cumsum(sizes, 0) - sizes
    room = (sizes[ref] - m + 1).to(torch.float64)
    start = firsts[ref] + (torch.rand(nq, device=_DEV, dtype=torch.float64, generator=g) * room).to(torch.int64)
    copied = _rand(g, nq) < case["sampled"]
    n_subs = torch.randint(0, case["subs"] + 1, (nq,), device=_DEV, generator=g) * copied
    has_n = _rand(g, nq) < case["with_n"]
    bases = torch.empty(int(offsets[-1]), dtype=torch.uint8, device=_DEV)
    step = max(1, (1 << 27) // m1)
    for a in range(0, nq, step):
        b = min(nq, a + step)
        lo, hi = int(offsets[a]), int(offsets[b])
        mm = m[a:b]

        def each(x):
            return torch.repeat_interleave(x[a:b], mm, output_size=hi - lo)

        j = torch.arange(lo, hi, device=_DEV) - each(offsets[:-1])
        rc = each(other)
        at = each(start) + torch.where(rc, each(m) - 1 - j, j)
        c = genomes.codes[at]
        c = torch.where(rc, 3 - c, c)
        c = torch.where(each(copied), c, _ints(g, 0, 4, hi - lo))
        for s in range(case["subs"]):
            q = torch.nonzero(n_subs[a:b] > s)[:, 0]
            p = offsets[a:b][q] - lo + (_rand(g, q.numel()) * mm[q]).to(torch.int64).clamp_(max=m1 - 1)
            p = torch.minimum(p, offsets[a + 1:b + 1][q] - lo - 1)
            c[p] = (c[p] + _ints(g, 1, 4, q.numel())) & 3
        c = _ascii(c)
        q = torch.nonzero(has_n[a:b])[:, 0]
        c[offsets[a:b][q] - lo + mm[q] // 2] = 78
        bases[lo:hi] = c
    q_ref = None
    if case["refs"] > 1 or case["strand"]:
        q_ref = torch.where(other, ref + sa.STRAND_BIT, ref)
        q_ref = torch.where(q_ref >= 1 << 31, q_ref - (1 << 32), q_ref).to(torch.int32)
    return bases, offsets, q_ref


def prepare(case, seed):
    g = torch.Generator(device=_DEV).manual_seed(int(seed) * 2 + 1)
    if case["kind"] == "build":
        _resident.clear()
        gc.collect()
        text = _to_ascii(_codes(g, case["n"], case["text"]))
        torch.cuda.empty_cache()
        return {"kind": "build", "text": text, "width": case["width"]}
    genomes = _genomes(case, int(seed) * 2)
    bases, offsets, q_ref = _queries(case, genomes, g)
    s = {"kind": case["kind"], "genomes": genomes, "bases": bases, "offsets": offsets, "q_ref": q_ref,
         "cap": case["cap"], "params": None}
    if case["strand"] or case["q_range"]:
        p = sa.sa_search_params()
        if case["strand"]:
            p.flags |= sa.SA_PARAM_STRAND_PER_QUERY
        if case["q_range"]:
            p.flags |= sa.SA_PARAM_Q_RANGE
            p.q_first, p.q_total = 0, bases.numel()
        s["params"] = p
    nq = case["nq"]
    room = max(4, nq * min(case["cap"], 32 if case["kind"] == "twocall" else 4))
    pos_type = torch.int32 if case["width"] == 32 else torch.int64
    if case["kind"] != "host":
        s["out"] = torch.zeros((nq, sa.RESULT_FIELDS), dtype=torch.int64, device=_DEV)
    if case["kind"] in ("locate", "twocall"):
        s["out_offsets"] = torch.zeros(nq + 1, dtype=torch.int64, device=_DEV)
        s["out_pos"] = torch.zeros(room, dtype=pos_type, device=_DEV)
    if case["kind"] == "host":
        for k in ("bases", "offsets", "q_ref"):
            if s[k] is not None:
                s[k] = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=True).copy_(s[k])
        s["out"] = torch.zeros((nq, sa.RESULT_FIELDS), dtype=torch.int64, pin_memory=True)
        s["out_offsets"] = torch.zeros(nq + 1, dtype=torch.int64, pin_memory=True)
        # the caller of a host batch is told when its positions do not fit: room for all
        s["out_pos"] = torch.zeros(max(4, nq * case["cap"]), dtype=pos_type, pin_memory=True)
    torch.cuda.empty_cache()
    return s


def run(s):
    if s["kind"] == "build":
        idx = sa.sa_build(s["text"], width=s["width"])
        out = idx.suffix_array()
        idx.free()
        return out
    refs = s["genomes"].indexes
    if s["kind"] == "search":
        return sa.sa_search_batch(refs, s["bases"], s["offsets"], q_ref=s["q_ref"], out=s["out"], params=s["params"])
    if s["kind"] == "twocall":
        res = sa.sa_search_batch(refs, s["bases"], s["offsets"], q_ref=s["q_ref"], out=s["out"], params=s["params"])
        offs, pos = sa.sa_locate(refs, res, s["cap"], q_ref=s["q_ref"], out_offsets=s["out_offsets"],
                                 out_pos=s["out_pos"])
        return res, offs, pos
    try:
        return sa.sa_search_locate(refs, s["bases"], s["offsets"], s["cap"], q_ref=s["q_ref"], out=s["out"],
                                   out_offsets=s["out_offsets"], out_pos=s["out_pos"], params=s["params"])
    except sa.SAError as e:
        # from host buffers the call also reports that some reads hold an N;
        # every result is there and those reads are marked
        if e.status != sa.SA_ERR_BASE:
            raise
        return s["out"], s["out_offsets"], s["out_pos"]


def exact(case, seed):
    """Every output is a whole number, which has one right value: nothing is rounded."""
    return None


def work(case):
    n, w = case["n"], case["width"] // 8
    if case["kind"] == "build":
        k = 1
        while k < 15 and 4 ** (k + 1) <= 3 * n:
            k += 1
        # the text in; packed text, suffix array, suffix records and k-mer
        # entries written once; the array read and written again by its copy
        return {"bytes": n + n / 4 + w * n + 32 * n + 64 * 4.0 ** k + 2 * w * n, "flops": 0}
    nq, mean = case["nq"], (case["m0"] + case["m1"]) / 2
    # bases and offsets in, one sector of the index per query, results out
    b = nq * (mean + 8 + 32 + 32) + (4 * nq if case["refs"] > 1 or case["strand"] else 0)
    if case["kind"] != "search":  # offsets, and about one position per copied query, read and written
        b += nq * (8 + case["sampled"] * 2 * w)
    return {"bytes": b, "flops": 0}
