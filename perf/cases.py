"""The workloads of this library whose speed counts, each through the public binding.

A case names a kind of work and its sizes; ``prepare`` makes what a user's program has in hand (strings, a grammar,
a context), ``run`` is one pass and returns all that it computes.  The strings are synthetic, made on the GPU: random
genomes and their variants (SNPs, indels, N-runs, repeat families) and Zipf-distributed text with copied blocks, with
the shapes of the benchmark's collections.

Kinds:
  compress  BuildGram over a collection on the device, and the grammar's VByte form in a device buffer (storing it)
  request   BuildGram over one string or a few in host memory; the roots and the packed form in host memory (serving)
  ingest    batches parsed one after another into a resident grammar, and its VByte form
  merge     two grammars arriving in VByte form, MergeGrams, and the result's VByte form (a step of a merge tree)
  expand    every string of a grammar expanded into a device buffer
  simplify  run-length rules and simplification of a grammar, and the result's host arrays
  codec     a column of 32-bit symbols to its VByte stream and back

Every output is a whole number or a byte, so it has one right value.  A result whose size depends on the strings is
returned in the buffer that a program keeps for it, whose rest stays zero.
"""
import collections
import math
import random

import numpy as np
import torch

from paper_2411_12439_gb300 import Context

HashFamily = collections.namedtuple("HashFamily", "levels m_bits a b c")
_P61 = (1 << 61) - 1


def hash_family(levels=64, m_bits=32):
    """The parameters that a program draws once and keeps for all its grammars."""
    r = random.Random(61)
    a, b, c = (np.array([r.randrange(1, _P61) for _ in range(levels)], dtype=np.uint64) for _ in range(3))
    return HashFamily(levels, m_bits, a, b, c)


# --------------------------------------------------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------------------------------------------------

def _dna(k, length, **kw):
    """k strings of about `length` bases, from `bases` random genomes.  `windows`: lengths spread over a factor of
    about ten instead of whole genomes.  `repeats`: copies of repeat families; `n_runs`: share of N-runs."""
    return dict({"k": k, "length": length, "bases": 1, "snp": 0.001, "indel": 0.0, "windows": False, "repeats": False,
                 "n_runs": 0.0, "text": False}, **kw)


def _text(k, length):
    return _dna(k, length, bases=0, snp=0.0, text=True)


def listed():
    return [
        # one short request of a serving loop: launches and latency only
        {"name": "request_20k", "kind": "request", **_dna(1, 20_011)},
        # a small collection of variants of one genome
        {"name": "compress_8x1M", "kind": "compress", "graph": False, **_dna(8, 1_000_000, indel=0.0001)},
        # a batch of bacterial genomes, built again and again as one CUDA graph
        {"name": "compress_64x5M_graph", "kind": "compress", "graph": True,
         **_dna(64, 5_000_000, bases=4, snp=0.01, indel=0.0002)},
        # byte text: a large alphabet and many distinct phrases
        {"name": "compress_text_32x2M", "kind": "compress", "graph": False, **_text(32, 2_000_003)},
        # many strings of very different lengths
        {"name": "compress_uneven_400x4M", "kind": "compress", "graph": False,
         **_dna(400, 4_000_000, bases=10, snp=0.015, indel=0.0007, windows=True)},
        # a few very long repetitive strings with N-runs: the benchmark's largest collection
        {"name": "compress_4x3100M", "kind": "compress", "graph": False,
         **_dna(4, 3_100_000_000, repeats=True, n_runs=0.01)},
        # a server's batches, parsed against the grammar they extend
        {"name": "ingest_6x12M", "kind": "ingest", "batches": 6, **_dna(48, 1_500_000, bases=3, snp=0.005, indel=0.0001, windows=True)},
        # a step of the merge tree over the parts of a collection
        {"name": "merge_2x16x5M", "kind": "merge", **_dna(32, 5_000_000, bases=2, snp=0.01, indel=0.0002)},
        # one short string read back
        {"name": "expand_20k", "kind": "expand", **_dna(1, 20_011)},
        # a collection of long strings read back
        {"name": "expand_4x200M", "kind": "expand", **_dna(4, 200_000_003, repeats=True, n_runs=0.01)},
        # the grammar made smaller for storage
        {"name": "simplify_16x2M", "kind": "simplify", **_dna(16, 2_000_000, bases=2, snp=0.005, n_runs=0.01)},
        # the plain codec over a column of a large grammar
        {"name": "codec_50M", "kind": "codec", "n": 50_000_003, "bits": 27},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _draw_strings(rng, least, most):
    """A collection of between `least` and `most` bytes in all."""
    total = _log(rng, least, most)
    k = min(_log(rng, 1, 600), max(1, total // 1000))
    length = total // k + rng.randrange(7)
    if rng.random() < 0.2 and total <= 100_000_000:
        return _text(k, length)
    return _dna(k, length, bases=min(k, _log(rng, 1, 12)), snp=rng.choice([0.001, 0.005, 0.01, 0.02]),
                indel=rng.choice([0.0, 0.0001, 0.0005]) if length < 20_000_000 else 0.0, windows=rng.random() < 0.4,
                repeats=length >= 1_000_000 and rng.random() < 0.3, n_runs=rng.choice([0.0, 0.0, 0.01]))


def draw(rng):
    kind = rng.choice(["compress", "compress", "compress", "request", "ingest", "merge", "expand", "simplify", "codec"])
    if kind == "compress":
        s = _draw_strings(rng, 50_000, 6_000_000_000)
        # a graph keeps the memory of all its rounds: for collections built again and again, not for the largest
        return {"kind": kind, "graph": rng.random() < 0.3 and s["k"] * s["length"] <= 500_000_000, **s}
    if kind == "request":
        return {"kind": kind, **_draw_strings(rng, 10_000, 20_000_000)}
    if kind == "ingest":
        s = _draw_strings(rng, 500_000, 200_000_000)
        return {"kind": kind, "batches": min(s["k"], rng.randrange(1, 9)), **s}
    if kind == "merge":
        s = _draw_strings(rng, 100_000, 400_000_000)
        return {"kind": kind, **dict(s, k=max(2, s["k"]))}
    if kind == "expand":
        s = _draw_strings(rng, 10_000, 800_000_000)
        return {"kind": kind, **dict(s, k=min(s["k"], 64))}
    if kind == "simplify":
        return {"kind": kind, **_draw_strings(rng, 100_000, 40_000_000)}
    return {"kind": "codec", "n": _log(rng, 1_000, 100_000_000), "bits": rng.randrange(8, 33)}


# --------------------------------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------------------------------

_CHUNK = 1 << 28
_N = 4  # code of the letter N; 0..3 are A, C, G, T


def _genome(c, n, g, r):
    """Codes of a random genome of n bases, with repeat families and N-runs."""
    x = torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda", generator=g)
    if c["repeats"]:
        # one mutated fragment of a repeat family in every cell of 3100 bases
        cell = 3100
        cells = n // cell
        fams = [torch.randint(0, 4, (int(w),), dtype=torch.uint8, device="cuda", generator=g)
                for w in np.geomspace(300, 3000, 10)]
        w = np.array([1.0 / len(f) for f in fams])
        table = torch.zeros((10, cell), dtype=torch.uint8, device="cuda")
        for i, f in enumerate(fams):
            table[i, :len(f)] = f
        size = torch.tensor([len(f) for f in fams], device="cuda")
        at = torch.arange(cell, device="cuda")
        for c0 in range(0, cells, 65536):
            m = min(65536, cells - c0)
            fam = torch.multinomial(torch.tensor(w / w.sum(), device="cuda"), m, replacement=True, generator=g)
            ln = (size[fam] * torch.rand(m, device="cuda", generator=g)).long().clamp_(min=100)
            view = x[c0 * cell:(c0 + m) * cell].view(m, cell)
            use = (at[None, :] < ln[:, None]) & (torch.rand((m, cell), device="cuda", generator=g) > 0.15)
            view.copy_(torch.where(use, table[fam], view))
    todo = int(c["n_runs"] * n)
    while todo > 0:
        run = min(int(math.exp(r.uniform(0.0, math.log(50_000)))), max(1, n // 4))
        at = r.randrange(0, n - run + 1)
        x[at:at + run] = _N
        todo -= run
    return x


def _variant(c, x, out, g):
    """x with SNPs (the letter N stays) into `out`."""
    for s in range(0, x.numel(), _CHUNK):
        y, o = x[s:s + _CHUNK], out[s:s + _CHUNK]
        hit = (torch.rand(y.numel(), device="cuda", generator=g) < c["snp"]) & (y != _N)
        new = (y + torch.randint(1, 4, (y.numel(),), dtype=torch.uint8, device="cuda", generator=g)) & 3
        o.copy_(torch.where(hit, new, y))


def _indels(c, x, g):
    """x with short insertions and deletions."""
    times = torch.ones(x.numel(), dtype=torch.int64, device="cuda")
    at = torch.rand(x.numel(), device="cuda", generator=g)
    times[at < c["indel"] / 2] = 0
    ins = (at >= c["indel"] / 2) & (at < c["indel"])
    times[ins] += torch.randint(1, 30, (int(ins.sum()),), device="cuda", generator=g)
    first = torch.cumsum(times, 0) - times
    src = torch.repeat_interleave(times)
    y = x[src]
    new = torch.randint(0, 4, (y.numel(),), dtype=torch.uint8, device="cuda", generator=g)
    return torch.where(torch.arange(y.numel(), device="cuda") == first[src], y, new)


def _text_of(n, g, r):
    p = torch.arange(1, 257, dtype=torch.float64, device="cuda") ** -1.1
    cdf = torch.cumsum(p / p.sum(), 0).float()
    perm = torch.randperm(256, device="cuda", generator=g).to(torch.uint8)
    x = perm[torch.searchsorted(cdf, torch.rand(n, device="cuda", generator=g)).clamp_(max=255)]
    todo = int(0.3 * n)
    while todo > 0 and n > 4096:
        size = r.randrange(1024, min(65536, n // 3) + 1)
        to = r.randrange(size, n - size + 1)
        at = r.randrange(0, to - size + 1)
        x[to:to + size] = x[at:at + size]
        todo -= size
    return x


def _strings(c, seed):
    """The collection: (uint8 tensor on the GPU, host offsets)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    k, length = c["k"], c["length"]
    if c["text"]:
        parts = [_text_of(k * length, g, r)]
        lens = [length] * k
    else:
        letters = torch.tensor(list(b"ACGTN"), dtype=torch.uint8, device="cuda")
        genome = [_genome(c, length * (3 if c["windows"] else 1), g, r) for _ in range(c["bases"])]
        lens, parts = [], []
        for j in range(k):
            x = genome[j % c["bases"]]
            if c["windows"]:
                n = min(x.numel(), max(2, int(length * math.exp(r.gauss(-0.18, 0.6)))))
                at = r.randrange(0, x.numel() - n + 1)
                x = x[at:at + n]
            y = torch.empty(x.numel(), dtype=torch.uint8, device="cuda")
            _variant(c, x, y, g)
            if c["indel"]:
                y = _indels(c, y, g)
            for s in range(0, y.numel(), _CHUNK):
                y[s:s + _CHUNK] = letters[y[s:s + _CHUNK].int()]
            parts.append(y)
            lens.append(y.numel())
        del genome
    offsets = np.zeros(k + 1, dtype=np.uint64)
    np.cumsum(np.array(lens, dtype=np.uint64), out=offsets[1:])
    data = torch.cat(parts) if len(parts) > 1 else parts[0]
    torch.cuda.synchronize()  # a context runs on a stream of its own
    return data, offsets


def _distinct(c):
    """(bases that no other string repeats, mutations): what the size of a grammar grows with."""
    n = c["k"] * c["length"]
    if c["text"]:
        return float(n), 0.0
    return min(n, c["bases"] * c["length"] * (3 if c["windows"] else 1)), n * (c["snp"] + c["indel"])


def _vbyte_bytes(c):
    """About the bytes of the collection's grammar in VByte form."""
    base, changed = _distinct(c)
    each = 3.0 if c["text"] else 1.3
    return min(each * base + 60.0 * changed, each * c["k"] * c["length"]) + 4096


def _most(c):
    """More bytes than the collection has with any seed."""
    return int(c["k"] * c["length"] * (3.0 if c["windows"] else 1.0 + 20 * c["indel"])) + 1000


# --------------------------------------------------------------------------------------------------------------------
# passes
# --------------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    ctx = Context(hash_family())
    s = {"kind": kind, "ctx": ctx}
    if kind == "codec":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        # the ranks of a grammar: widths spread evenly up to that of the largest level
        width = torch.randint(1, case["bits"] + 1, (n,), device="cuda", generator=g)
        s["values"] = (torch.randint(0, 1 << 32, (n,), device="cuda", generator=g) >> (32 - width)).to(torch.int32)
        s["stream"] = torch.zeros(5 * n, dtype=torch.uint8, device="cuda")
        s["decoded"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        return s
    data, offsets = _strings(case, seed)
    k, n = case["k"], int(offsets[-1])

    def form():  # a buffer that the grammar's VByte form fits in
        return torch.zeros(int(1.5 * _vbyte_bytes(case) * (3 if case["windows"] else 1)) + (1 << 18),
                           dtype=torch.uint8, device="cuda")

    if kind == "compress":
        ctx.set_graph(case["graph"])
        s.update(data=data, offsets=offsets, out=form())
    elif kind == "request":
        s.update(data=data.cpu().pin_memory(), offsets=offsets,
                 out=torch.zeros((1 << 20) + (16 if case["text"] else 6) * _most(case), dtype=torch.uint8).pin_memory())
    elif kind == "ingest":
        cut = [k * b // case["batches"] for b in range(case["batches"] + 1)]
        s["batches"] = [(data[int(offsets[a]):int(offsets[b])].clone(), offsets[a:b + 1] - offsets[a])
                        for a, b in zip(cut, cut[1:])]
        s["out"] = form()
    elif kind == "merge":
        half = k // 2
        s["parts"] = []
        for a, b in ((0, half), (half, k)):
            gr = ctx.build(data[int(offsets[a]):int(offsets[b])], offsets[a:b + 1] - offsets[a])
            s["parts"].append(gr.export_vbyte(device=True))
            gr.free()
        s["out"] = form()
    else:
        s["grammar"] = ctx.build(data, offsets)
        if kind == "expand":
            s.update(offsets=[int(x) for x in offsets], out=torch.zeros(_most(case), dtype=torch.uint8, device="cuda"))
        else:  # where the program keeps the result: more than any seed's
            size = int(0.5 * _vbyte_bytes(case) * (3 if case["windows"] else 1)) + (1 << 16)
            s["kept"] = {"kind": np.zeros(size, np.uint8), "rhs_off": np.zeros(size, np.int64),
                         "rhs": np.zeros(size, np.int32), "c": np.zeros(k, np.int32)}
    return s


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "compress":
        g = ctx.build(state["data"], state["offsets"])
        g.export_vbyte(out=state["out"])
        g.free()
        return state["out"]
    if kind == "request":
        g = ctx.build(state["data"], state["offsets"])
        level, rank, fingerprint = g.roots()
        g.export_packed(out=state["out"])
        g.free()
        return {"level": level, "rank": rank, "fingerprint": fingerprint, "packed": state["out"]}
    if kind == "ingest":
        none = np.zeros(0, dtype=np.uint32)
        g = ctx.import_grammar({"levels": [], "c_level": none, "c_rank": none})
        for data, offsets in state["batches"]:
            ctx.build_into(g, data, offsets)
        level, rank, fingerprint = g.roots()
        g.export_vbyte(out=state["out"])
        g.free()
        return {"level": level, "rank": rank, "fingerprint": fingerprint, "vbyte": state["out"]}
    if kind == "merge":
        a, b = (ctx.import_vbyte(p) for p in state["parts"])
        ctx.merge(a, b)
        a.export_vbyte(out=state["out"])
        a.free()
        b.free()
        return state["out"]
    if kind == "expand":
        g, off, out = state["grammar"], state["offsets"], state["out"]
        for j in range(len(off) - 1):
            g.decompress(j, out=out[off[j]:off[j + 1]])
        return out
    if kind == "simplify":
        pp = ctx.postprocess(state["grammar"])
        out, kept = pp.stats(), state["kept"]
        for name, x in pp.export().items():
            kept[name][:x.shape[0]] = x.view(kept[name].dtype)
        pp.free()
        return {**out, **kept}
    stream = ctx.vbyte_encode(state["values"], out=state["stream"])
    ctx.vbyte_decode(stream, state["values"].numel(), out=state["decoded"])
    return {"bytes": stream.numel(), "stream": state["stream"], "decoded": state["decoded"]}


def work(case):
    """Bytes that a pass cannot do without: its input read and its output written, once each.  The sizes of grammars
    are estimates from the collection's make-up.  The path has no floating-point work."""
    kind = case["kind"]
    if kind == "codec":
        stream = case["n"] * sum((w + 6) // 7 for w in range(1, case["bits"] + 1)) / case["bits"]
        return {"bytes": 2 * (4 * case["n"] + stream), "flops": 0}
    n, vb = case["k"] * case["length"], _vbyte_bytes(case)
    moved = {"compress": n + vb, "request": n + 2.0 * vb, "ingest": n + vb, "merge": 2.2 * vb, "expand": n + vb,
             "simplify": 3.0 * vb}[kind]
    return {"bytes": moved, "flops": 0}


def exact(case, seed):
    """No output is a rounded number: all are compared for equality."""
    return None
