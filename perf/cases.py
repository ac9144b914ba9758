"""Timed cases of the index: what programs that use it call, over the range of
sizes they call it with.

An index holds K sets; it is filled by `Rambo.insert` and asked by
`Rambo.query_into` (arrays on the device), `Rambo.query` (arrays in host
memory) or a `Plan` (a captured query for a server's batches).  A pass of a
case is one such call, its answers kept in buffers of the program's own, or,
for the cases that fill an index, an insert followed by the lookups that read
it back.  Collections are synthetic with the shapes of `synth.workloads`
(genomes sharing Zipf-popular chunks, documents over a Zipf vocabulary, lone
k-mers), made on the GPU from the seed.

Every output is a set ID or an offset, so results are whole numbers that have
to be equal; nothing here is a rounded value.
"""
import math

import numpy as np
import torch

from paper_1910_02611_gb300 import Plan, Rambo

CHUNK = 1000  # bases of a genome's chunk
CANONICAL, SKIP_N = 0x100, 0x200  # flags of the k-mer length (include/rambo.h)

_DEFAULTS = dict(
    corpus="documents",  # documents: sets of terms; genomes: DNA whose k-mers are the keys; kmers: sets of lone 31-mers
    K=1000, B=32, R=4, m=1 << 16, eta=2,
    vocab=1_000_000, tokens=500,  # documents: vocabulary, mean tokens of one (repeats are inserted too)
    chunks=100, pool=10_000,  # genomes: chunks of one (half of them from a shared pool of `pool`)
    op="query",  # query: query_into or (host) query; plan: a captured Plan; insert: Rambo.insert, then a query
    host=False,  # inputs and answers in host memory
    insert=0,  # op insert: sets inserted by a pass (the index holds the others already)
    n=1,  # queries of a pass
    terms_lo=1, terms_hi=5,  # terms of a key query
    len_lo=100, len_hi=1000, median=0,  # bases of a DNA query: uniform, or lognormal (sigma 1) around a median
    subst=0.02,  # highest share of substituted bases of a DNA query
    k=31, canonical=False, skip_n=False,
)


def _case(name=None, **kw):
    c = dict(_DEFAULTS)
    c.update(kw)
    if name:
        c["name"] = name
    return c


# the four collections of the benchmark, and two of the paper's layouts beside them
_TINY = dict(corpus="kmers", K=100, B=10, R=3, m=1 << 20, eta=2, tokens=10_000, terms_lo=1, terms_hi=1)
_GENOME = dict(corpus="genomes", K=2000, B=64, R=6, m=1 << 27, eta=2, chunks=1000)
_UNEVEN = dict(corpus="genomes", K=10_000, B=128, R=8, m=1 << 26, eta=2, chunks=200)
_DOCUMENT = dict(corpus="documents", K=100_000, B=320, R=8, m=1 << 25, eta=3, tokens=700)
_ABSTRACTS = dict(corpus="documents", K=500_000, B=1000, R=6, m=1 << 22, eta=2, tokens=200)
_WIDE = dict(corpus="documents", K=100_000, B=20_000, R=4, m=1 << 16, eta=2, tokens=700)


def listed():
    return [
        # a search box: one query of three terms, asked and answered in host memory
        _case("one_lookup", K=10_000, B=100, R=4, m=1 << 22, eta=3, host=True, n=1, terms_lo=3, terms_hi=3),
        # k-mer screening against a small panel: 10^4 single 31-mers, an index that fits L2
        _case("tiny_kmers", n=10_000, **_TINY),
        # a search server's slot: what arrived meanwhile (16 queries of 1-5 terms) through a captured plan
        _case("serve_terms", op="plan", host=True, n=16, **_DOCUMENT),
        # reads and contigs against 2000 genomes: the paper's sequence search
        _case("genome_reads", n=100_000, **_GENOME),
        # the largest query batch: 10^6 sequences of very uneven length
        _case("uneven_reads", n=1_000_000, median=300, len_lo=31, len_hi=10_000, **_UNEVEN),
        # a command-line search: reads in pinned host memory, both strands, answers to host memory
        _case("reads_host", corpus="genomes", K=2000, B=64, R=6, m=1 << 24, eta=2, chunks=125, host=True, n=100_000,
              canonical=True),
        # sequencer output: short reads with unresolved bases, both strands, k = 21, an index of odd sizes
        _case("short_reads_n", corpus="genomes", K=500, B=100, R=5, m=1 << 23, eta=3, chunks=400, n=200_000, len_lo=100,
              len_hi=251, subst=0.01, k=21, canonical=True, skip_n=True),
        # document search in bulk: conjunctive queries whose terms follow the corpus, so answers are long
        _case("documents", n=100_000, **_DOCUMENT),
        # a larger collection of short documents (more set IDs than a per-query bitmap of shared memory holds)
        _case("abstracts", n=10_000, **_ABSTRACTS),
        # the paper's web index (B = 2*10^4, R = 4): few documents a cell, rows of 2.5 KB
        _case("web_wide", n=20_000, **_WIDE),
        # building an index from DNA (2*10^9 bases), and 10^6 k-mer lookups that read it back
        _case("build_genomes", op="insert", insert=2000, n=1_000_000, len_lo=31, len_hi=31, subst=0.0, **_GENOME),
        # a collection that grows while it is searched: 100 documents from host memory, then 256 lookups
        _case("stream_documents", op="insert", insert=100, host=True, n=256, **_DOCUMENT),
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _filter_bits(keys, eta, lo, hi):
    """Bits of a Bloom filter that `keys` keys of eta hashes fill to a fifth or a third."""
    m = 1 << lo
    while m < 3 * keys * eta and m < 1 << hi:
        m <<= 1
    return m


def draw(rng):
    kind = rng.choice(("documents", "documents", "reads", "reads", "wide", "kmers", "insert"))
    if kind in ("documents", "wide", "insert"):
        wide = kind == "wide"
        K = _between(rng, 10_000, 130_000) if wide else _between(rng, 1000, 300_000)
        B = rng.randint(5000, 50_000) if wide else max(16, min(1000, int(math.sqrt(K) * rng.uniform(0.6, 2.0))))
        R, eta, tokens = rng.randint(3, 6 if wide else 8), rng.randint(1, 3 if wide else 4), _between(rng, 50, 700)
        c = _case(corpus="documents", K=K, B=B, R=R, eta=eta, tokens=tokens,
                  m=_filter_bits(0.75 * K * tokens / B, eta, 11 if wide else 14, 16 if wide else 23))
        c["terms_hi"] = rng.randint(1, 8)
        c["host"] = rng.random() < 0.3
        c["n"] = _between(rng, 1, 20_000 if wide else max(2, min(100_000, int(8e9 / K))))
        if kind == "insert":
            c.update(op="insert", insert=_between(rng, 1, min(2000, K // 2)), n=_between(rng, 16, 1024))
        elif rng.random() < 0.3:
            c.update(op="plan", host=True, n=_between(rng, 1, 256))
        return c
    if kind == "kmers":
        K = _between(rng, 20, 1000)
        B, eta, tokens = rng.randint(5, 100), rng.randint(1, 4), _between(rng, 1000, 20_000)
        return _case(corpus="kmers", K=K, B=B, R=rng.randint(2, 8), eta=eta, tokens=tokens,
                     m=_filter_bits(K * tokens / B, eta, 14, 24), n=_between(rng, 16, 300_000), terms_lo=1,
                     terms_hi=rng.randint(1, 4), host=rng.random() < 0.5)
    K = _between(rng, 50, 10_000)
    B, R, eta = rng.randint(10, 200), rng.randint(3, 8), rng.randint(1, 3)
    chunks = _between(rng, 10, max(12, min(1000, 500_000 // K)))
    median = rng.choice((0, 0, 200, 400))
    lo = rng.randint(80, 200)
    hi = 8000 if median else lo + rng.randint(1, 1500)
    mean = 1.6 * median if median else (lo + hi) / 2
    c = _case(corpus="genomes", K=K, B=B, R=R, eta=eta, chunks=chunks, m=_filter_bits(K * chunks * CHUNK * 0.75 / B, eta, 14, 25),
              n=_between(rng, 32, min(300_000, int(1.5e8 / mean))), len_lo=lo, len_hi=hi, median=median,
              subst=rng.choice((0.0, 0.01, 0.02)), k=rng.choice((15, 21, 31, 31, 32)), canonical=rng.random() < 0.4,
              skip_n=rng.random() < 0.25, host=rng.random() < 0.3)
    if rng.random() < 0.2:
        c.update(op="plan", host=True, n=_between(rng, 32, 256))
    return c


# ----------------------------------------------------------------------------
# collections and queries, on the GPU


def _bases(g, shape):
    """Random ASCII bases."""
    x = torch.randint(0, 4, shape, dtype=torch.uint8, device="cuda", generator=g)
    return 65 + 2 * x + 2 * (x == 2).to(torch.uint8) + 13 * (x == 3).to(torch.uint8)  # A C G T


def _genomes(c, g):
    """[K, chunks * CHUNK] bases: half of a genome's chunks from a shared pool by Zipf(1.1) popularity, half its own."""
    K, C = c["K"], c["chunks"]
    P = max(C, c["pool"])
    shared = C // 2
    pool = _bases(g, (P, CHUNK))
    logw = -1.1 * torch.log(torch.arange(1, P + 1, device="cuda", dtype=torch.float32))
    data = torch.empty((K, C, CHUNK), dtype=torch.uint8, device="cuda")
    step = max(1, min(K, (1 << 27) // (C * CHUNK), (1 << 26) // P))
    for a in range(0, K, step):
        b = min(K, a + step)
        u = torch.rand((b - a, P), device="cuda", generator=g).clamp_(1e-9, 1 - 1e-7)
        picks = (logw - torch.log(-torch.log(u))).topk(shared, dim=1).indices if shared else None
        own = _bases(g, (b - a, C - shared, CHUNK))
        chunks = torch.cat([pool[picks], own], 1) if shared else own
        order = torch.rand((b - a, C), device="cuda", generator=g).argsort(dim=1)
        data[a:b] = chunks[torch.arange(b - a, device="cuda")[:, None], order]
    data = data.view(K, C * CHUNK)
    if c["skip_n"]:  # assemblies have gaps: a run of unresolved bases in every genome
        data[:, 100:150] = ord("N")
    return data


def _reads(c, genomes, g):
    """(bases, offsets): substrings of random genomes, each with its own share of substituted bases."""
    n, L = c["n"], genomes.shape[1]
    if c["median"]:
        lens = torch.empty(n, device="cuda").normal_(math.log(c["median"]), 1.0, generator=g).exp_().round_()
    else:
        lens = torch.randint(c["len_lo"], c["len_hi"] + 1, (n,), device="cuda", generator=g)
    lo = max(c["len_lo"], 2 * c["k"] + 1 if c["skip_n"] else c["k"])
    lens = lens.long().clamp_(lo, max(lo, min(c["len_hi"], L - 300)))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    which = torch.randint(0, genomes.shape[0], (n,), device="cuda", generator=g)
    start = (torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * (L - 200 - lens + 1)).long() + 200
    at = torch.repeat_interleave(which * L + start - off[:-1], lens)
    at += torch.arange(at.numel(), device="cuda")
    data = genomes.reshape(-1)[at]
    del at
    if c["subst"]:
        rate = torch.rand(n, device="cuda", generator=g) * c["subst"]
        hit = (torch.rand(data.numel(), device="cuda", generator=g) < torch.repeat_interleave(rate, lens)).nonzero().view(-1)
        code = torch.zeros(256, dtype=torch.int64, device="cuda")
        code[[65, 67, 71, 84]] = torch.arange(4, device="cuda")
        letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
        turn = torch.randint(1, 4, (hit.numel(),), device="cuda", generator=g)
        data[hit] = letters[(code[data[hit].long()] + turn) & 3]
    if c["skip_n"]:  # one unresolved base in every tenth read
        some = torch.arange(0, n, 10, device="cuda")
        at = off[some] + (torch.rand(some.numel(), device="cuda", generator=g) * lens[some]).long().clamp_(max=c["len_hi"])
        data[torch.minimum(at, off[some + 1] - 1)] = ord("N")
    return data, off


def _any_keys(g, n):
    return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device="cuda", generator=g)


def _documents(c, g):
    """(terms, offsets, share of each vocabulary entry, keys): lognormal lengths, terms by Zipf(1) popularity."""
    V = c["vocab"]
    vocab = _any_keys(g, V)
    w = 1.0 / torch.arange(1, V + 1, device="cuda", dtype=torch.float64)
    cdf = torch.cumsum(w, 0) / w.sum()
    lens = torch.empty(c["K"], device="cuda").normal_(math.log(c["tokens"]) - 0.5, 1.0, generator=g).exp_()
    lens = lens.round_().long().clamp_(1, 100 * c["tokens"])
    off = torch.zeros(c["K"] + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    total = int(off[-1])
    terms = torch.empty(total, dtype=torch.int64, device="cuda")
    for a in range(0, total, 1 << 26):
        u = torch.rand(min(1 << 26, total - a), device="cuda", dtype=torch.float64, generator=g)
        terms[a : a + u.numel()] = vocab[torch.searchsorted(cdf, u).clamp_(max=V - 1)]
    seen = 1.0 - torch.exp(-c["tokens"] * w / w.sum())  # share of the documents that hold a term
    return terms, off, torch.cumsum(seen, 0) / seen.sum(), vocab


def _term_queries(c, cdf, vocab, g):
    n = c["n"]
    nt = torch.randint(c["terms_lo"], c["terms_hi"] + 1, (n,), device="cuda", generator=g)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(nt, 0, out=off[1:])
    u = torch.rand(int(off[-1]), device="cuda", dtype=torch.float64, generator=g)
    return vocab[torch.searchsorted(cdf, u).clamp_(max=vocab.numel() - 1)], off


def _kmer_sets(c, g):
    K, s = c["K"], c["tokens"]
    return (torch.randint(0, 1 << 62, (K * s,), dtype=torch.int64, device="cuda", generator=g),
            torch.arange(0, (K + 1) * s, s, device="cuda"))


def _kmer_queries(c, sets, g):
    """Half of the queries hold k-mers of one set, half hold fresh ones."""
    n, s = c["n"], c["tokens"]
    nt = torch.randint(c["terms_lo"], c["terms_hi"] + 1, (n,), device="cuda", generator=g)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(nt, 0, out=off[1:])
    total = int(off[-1])
    which = torch.repeat_interleave(torch.randint(0, c["K"], (n,), device="cuda", generator=g), nt)
    member = sets[which * s + torch.randint(0, s, (total,), device="cuda", generator=g)]
    fresh = torch.randint(0, 1 << 62, (total,), dtype=torch.int64, device="cuda", generator=g)
    known = torch.repeat_interleave(torch.rand(n, device="cuda", generator=g) < 0.5, nt)
    return torch.where(known, member, fresh), off


def _to_host(t, kind):
    """The same values in pinned host memory, as numpy."""
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    a = h.numpy()
    return a if kind == "seq" and t.dtype == torch.uint8 else a.view(np.uint64)


def prepare(case, seed):
    c = dict(_DEFAULTS)
    c.update(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = "seq" if c["corpus"] == "genomes" else "keys"
    k = c["k"] | (CANONICAL if c["canonical"] else 0) | (SKIP_N if c["skip_n"] else 0)
    K = c["K"]
    if c["corpus"] == "genomes":
        genomes = _genomes(c, g)
        data, off = genomes.view(-1), torch.arange(0, (K + 1) * genomes.shape[1], genomes.shape[1], device="cuda")
        q, qo = _reads(c, genomes, g)
    elif c["corpus"] == "documents":
        data, off, cdf, vocab = _documents(c, g)
        q, qo = _term_queries(c, cdf, vocab, g)
    else:
        data, off = _kmer_sets(c, g)
        q, qo = _kmer_queries(c, data, g)
    ids = torch.arange(K, device="cuda")
    index = Rambo(K, c["B"], c["R"], c["m"], c["eta"], 42)
    s = {"index": index, "kind": kind, "k": k, "q": q, "qo": qo, "new": None, "plan": None, "host": c["host"]}
    old = K - c["insert"]
    if old:
        index.insert(ids[:old], data, off[: old + 1], kind=kind, k=k)
    if c["insert"]:
        new = data[int(off[old]) :].clone() if old else data
        s["new"] = (ids[old:].clone(), new, off[old:] - off[old])
    if c["host"]:
        s["q"], s["qo"] = _to_host(q, kind), _to_host(qo, "keys")
        if s["new"]:
            i, d, o = s["new"]
            s["new"] = (_to_host(i, "keys"), _to_host(d, kind), _to_host(o, "keys"))
    # room for the answers: any answer of a small batch, two fifths of all sets for a large one's mean
    room = c["n"] * K if c["n"] * K <= 10**8 else c["n"] * K * 2 // 5
    if c["op"] == "plan":
        s["plan"] = Plan(index, kind, c["n"], max(1, int(qo[-1])), room, k)
    if c["host"]:
        s["ids"] = np.zeros(room, np.uint32)
    else:
        s["ids"] = torch.zeros(room, dtype=torch.int32, device="cuda")
        s["off"] = torch.zeros(c["n"] + 1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    index, kind, k = s["index"], s["kind"], s["k"]
    if s["new"] is not None:
        ids, data, off = s["new"]
        index.insert(ids, data, off, kind=kind, k=k)
    if not s["host"]:
        index.query_into(s["q"], s["qo"], s["ids"], s["off"], kind=kind, k=k)
        return s["ids"], s["off"]
    if s["plan"] is not None:
        s["plan"].launch_host(s["q"], s["qo"])
        ids, off = s["plan"].wait(to_host=True)
    else:
        ids, off = index.query(s["q"], s["qo"], kind=kind, k=k, copy=False)
    s["ids"][: ids.size] = ids
    return s["ids"].view(np.int32), off.astype(np.int64)


def exact(case, seed):
    """Nothing to compare in 64 bits: every output is a whole number (a set ID or an offset)."""
    return None


# ----------------------------------------------------------------------------
# what a pass cannot do without


def _mean_answer(c):
    """Mean number of sets in an answer, from the collection's distribution (false positives left out)."""
    if c["corpus"] == "kmers":
        return 0.5
    if c["corpus"] == "documents":
        w = 1.0 / np.arange(1, c["vocab"] + 1)
        seen = 1.0 - np.exp(-c["tokens"] * w / w.sum())
        one = float((seen * seen).sum() / seen.sum())  # share of documents holding a query's term
        t = np.arange(c["terms_lo"], c["terms_hi"] + 1)
        return c["K"] * float((one**t).mean())
    mean = min(c["len_hi"], 1.65 * c["median"]) if c["median"] else (c["len_lo"] + c["len_hi"]) / 2
    return _whole_share(c, mean) * max(1.0, 0.5 * c["K"] * (c["chunks"] // 2) / max(c["chunks"], c["pool"]))


def _whole_share(c, length):
    """Share of DNA queries of that length without a substituted base."""
    if not c["subst"]:
        return 1.0
    x = length * c["subst"]
    return (1.0 - math.exp(-x)) / x


def work(case):
    c = dict(_DEFAULTS)
    c.update(case)
    row = -(-(-(-c["B"] // 32) * 4) // 32) * 32  # bytes of a row, in whole sectors
    index = float(c["R"]) * c["m"] * max(4 * -(-c["B"] // 32), 4)
    probes = c["R"] * c["eta"]
    if c["corpus"] == "genomes":
        # a query whose k-mers are all present reads R * eta rows for each; another is settled by one absent k-mer
        grid = np.exp(math.log(c["median"]) + np.linspace(-3, 3, 61)) if c["median"] else np.linspace(c["len_lo"], c["len_hi"], 61)
        p = np.exp(-np.linspace(-3, 3, 61) ** 2 / 2) if c["median"] else np.ones(61)
        grid, p = np.clip(grid, max(c["len_lo"], c["k"]), c["len_hi"]), p / p.sum()
        whole = np.array([_whole_share(c, x) for x in grid])
        rows = c["n"] * float((p * (whole * (grid - c["k"] + 1) * probes + (1 - whole) * c["eta"])).sum())
        asked = c["n"] * float((p * grid).sum())
    else:
        terms = c["n"] * (c["terms_lo"] + c["terms_hi"]) / 2
        whole = 0.5 if c["corpus"] == "kmers" else 1.0
        rows = terms * (whole * probes + (1 - whole) * c["eta"])
        asked = 8 * terms
    moved = asked + 16 * (c["n"] + 1) + min(rows * row, index) + 4 * c["n"] * _mean_answer(c)
    if c["op"] == "insert":
        keys = c["insert"] * (c["chunks"] * CHUNK if c["corpus"] == "genomes" else c["tokens"])
        # the sets are read once, and every sector that holds one of their bits is read and written at most once
        moved += keys * (1 if c["corpus"] == "genomes" else 8) + 2 * min(index, 32.0 * keys * probes)
    return {"bytes": moved, "flops": 0.0}
