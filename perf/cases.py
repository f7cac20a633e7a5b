"""Performance cases of the spliced protein-to-genome aligner.

Each case is one call (or one short sequence of calls) of the library's
public entry points on synthetic inputs shaped like the benchmark's
workloads: proteins planted in genomic regions with substitutions,
frameshift indels and GT...AG introns.  A case's sizes (protein lengths,
introns, flanks, strands) follow from the case alone; the sequences follow
from the seed.

Kinds of case:
  align    mp_dp_align_batch from host sequences, or, with resident, one run
           of an uploaded batch and the download of its results
  regions  mp_dp_align_batch over windows of one genome (several per
           protein), with pseudogene-aware rescoring when asked for
  serve    a burst of mp_dp_submit requests, each polled for its result
  map      mp_index_build of a genome, then mp_index_chain of a few proteins
  chain    mp_index_chain of many proteins against an index kept by the caller
  refine   mp_chain_refine over candidate regions
"""
from __future__ import annotations

import ctypes

import numpy as np

import paper_2210_08052_gb300 as mp

AA = np.frombuffer(b"ARNDCQEGHILKMFPSTWYV", dtype=np.uint8)
# background amino-acid frequencies (Robinson & Robinson 1991), in that order
FREQ = np.array([0.07805, 0.05129, 0.04487, 0.05364, 0.01925, 0.04264, 0.06295, 0.07377, 0.02199, 0.05142,
                 0.09019, 0.05744, 0.02243, 0.03856, 0.05203, 0.07120, 0.05841, 0.01330, 0.03216, 0.06441])
CODON_AA = "KNKNTTTTRSRSIIMIQHQHPPPPRRRRLLLLEDEDAAAAGGGGVVVV*Y*YSSSS*CWCLFLF"      # codons in A, C, G, T order
CODONS = [[c for c in range(64) if CODON_AA[c] == a] for a in AA.tobytes().decode()]
N_SYN = np.array([len(c) for c in CODONS])
SYN = np.array([(c * 6)[:6] for c in CODONS])
ACGT = np.frombuffer(b"ACGT", dtype=np.uint8)
GC40 = np.frombuffer(b"AAACCGGTTT", dtype=np.uint8)                                  # 40% GC
COMP = np.arange(256, dtype=np.uint8)
COMP[ACGT] = ACGT[::-1]


def listed():
    return [
        # one gene looked at by hand: the smallest call, latency and launches count
        dict(name="align_one", kind="align", mix="one", n=1, mode=0, resident=False, profile=False, shape=1),
        # a gene family against its candidate loci, sequences from the host
        dict(name="align_64", kind="align", mix="genes", n=64, mode=0, resident=False, profile=False, shape=2),
        # the benchmark's batch, its sequences kept on the device
        dict(name="resident_4096", kind="align", mix="genes", n=4096, mode=0, resident=True, profile=False, shape=3),
        # a proteome of very uneven lengths with decoys and long introns: more traceback than the budget, in waves
        dict(name="uneven_1500", kind="align", mix="uneven", n=1500, mode=0, resident=False, profile=False, shape=4),
        # closing the gaps between anchors (global mode; the draws take the extension mode too)
        dict(name="global_512", kind="align", mix="genes", n=512, mode=1, resident=False, profile=False, shape=5),
        # giant proteins of close relatives, whose scores leave 16 bits
        dict(name="long_8", kind="align", mix="long", n=8, mode=0, resident=False, profile=False, shape=6),
        # family profiles with position-specific scores and gap costs
        dict(name="profile_128", kind="align", mix="genes", n=128, mode=0, resident=False, profile=True, shape=7),
        # candidate windows of one genome, three per protein, pseudogene-aware scores
        dict(name="regions_3000", kind="regions", n=3000, genome=20_000_000, rescore=True, shape=8),
        # requests of a serving loop that arrive together
        dict(name="serve_32", kind="serve", n=32, shape=9),
        # a new genome: its index, and the chains of the few proteins asked for
        dict(name="map_50mb", kind="map", n=64, genome=50_000_000, shape=10),
        # a proteome against an index that is kept
        dict(name="chain_4000", kind="chain", n=4000, genome=50_000_000, shape=11),
        # second chaining round of the candidate regions
        dict(name="refine_6000", kind="refine", n=6000, shape=12),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    shape = rng.randrange(1 << 30)
    kind = rng.choice(["align", "align", "align", "regions", "serve", "map", "chain", "refine"])
    if kind == "align":
        mix = rng.choice(["one", "genes", "genes", "uneven", "long"])
        n = {"one": 1, "genes": _log(rng, 1, 4096), "uneven": _log(rng, 1, 1500), "long": rng.randint(1, 8)}[mix]
        profile = mix == "genes" and n <= 256 and rng.random() < 0.3
        return dict(kind=kind, mix=mix, n=n, mode=rng.choice([0, 0, 1, 2]), resident=rng.random() < 0.5,
                    profile=profile, shape=shape)
    if kind == "regions":
        return dict(kind=kind, n=_log(rng, 30, 3000), genome=_log(rng, 1_000_000, 20_000_000),
                    rescore=rng.random() < 0.5, shape=shape)
    if kind == "serve":
        return dict(kind=kind, n=_log(rng, 1, 64), shape=shape)
    if kind == "map":
        return dict(kind=kind, n=_log(rng, 1, 64), genome=_log(rng, 300_000, 50_000_000), shape=shape)
    if kind == "chain":
        return dict(kind=kind, n=_log(rng, 16, 4000), genome=_log(rng, 1_000_000, 50_000_000), shape=shape)
    return dict(kind=kind, n=_log(rng, 1, 6000), shape=shape)


# ------------------------------------------------------------------- sizes
def _lognormal(r, median, sigma, lo, hi, n):
    return np.clip(np.round(np.exp(r.normal(np.log(median), sigma, n))), lo, hi).astype(np.int64)


def _genes(r, mix, n):
    """Per pair: protein length, intron lengths, flank, substitution rate, frameshift indels (+1 or -1 base),
    strand and whether only its score is wanted."""
    out = []
    for _ in range(n):
        if mix == "one":
            out.append((120, [150, 400], 100, 0.15, [1], 1, False))
            continue
        if mix == "uneven":
            m = int(round(20 * 250 ** r.random()))
        elif mix == "long":
            m = int(r.integers(6500, 9000))
        else:
            m = int(_lognormal(r, 350, 0.75, 50, 2000, 1)[0])
        introns = _lognormal(r, 800, 1.0, 60, 20000, min(int(r.poisson(3)), 8)).tolist()
        if mix == "uneven" and r.random() < 0.02:
            introns.append(int(r.integers(20_000, 100_000)))
        rate = r.uniform(0.0, 0.04) if mix == "long" else r.uniform(0.1, 0.4)
        shifts = r.choice([-1, 1], size=int(r.integers(0, 4))).tolist()
        out.append((m, introns, 1000, rate, shifts, 1 if r.random() < 0.5 else -1,
                    mix == "uneven" and r.random() < 0.05))
    return out


def _nt_len(g):
    return 3 * g[0] + sum(g[1]) + 2 * g[2] + sum(g[4])


def _region_sizes(case):
    """Planted genes and, for each of them, where its three windows lie in the genome."""
    r = np.random.default_rng(case["shape"])
    per = 3
    genes = _genes(r, "genes", -(-case["n"] // per))
    pitch = case["genome"] // (len(genes) + 1)
    spans = [min(_nt_len(g) - 2000, case["genome"] - 4000) for g in genes]
    at = [min(1000 + k * pitch, case["genome"] - s - 1000) for k, s in enumerate(spans)]
    win = []
    for k, s in enumerate(spans):
        win.append((k, at[k] - 1000, s + 2000, genes[k][5]))
        for _ in range(per - 1):
            win.append((k, int(r.integers(0, case["genome"] - s - 2000 + 1)), s + 2000, 1 if r.random() < 0.5 else -1))
    return genes, at, spans, win[:case["n"]]


def _proteome(case):
    """Protein lengths of a map or chain case and how many of them have a gene in the genome."""
    r = np.random.default_rng(case["shape"])
    lens = _lognormal(r, 350, 0.75, 50, 2000, case["n"])
    return lens, max(1, case["n"] // 10)


# --------------------------------------------------------------- sequences
def _protein(rng, m):
    return rng.choice(20, size=m, p=FREQ)


def _coding(rng, prot, rate):
    """A coding sequence of the protein with a fraction of its residues substituted."""
    p = np.where(rng.random(len(prot)) < rate, rng.integers(0, 20, len(prot)), prot)
    c = SYN[p, (rng.random(len(p)) * N_SYN[p]).astype(np.int64)]
    return ACGT[np.stack([c >> 4, (c >> 2) & 3, c & 3], axis=1).reshape(-1)]


def _spliced(rng, prot, gene):
    """The gene's exons, introns and frameshifts, without flanks."""
    m, introns, _, rate, shifts, _, _ = gene
    cds = _coding(rng, prot, rate)
    for s in shifts:
        x = int(rng.integers(1, len(cds) - 1))
        cds = np.insert(cds, x, ACGT[rng.integers(0, 4)]) if s > 0 else np.delete(cds, x)
    parts, last = [], 0
    for x, n in zip(sorted(rng.integers(1, len(cds), len(introns)).tolist()), introns):
        intron = GC40[rng.integers(0, 10, n)]
        intron[:3] = np.frombuffer(b"GTA", dtype=np.uint8)
        intron[-3:] = np.frombuffer(b"CAG", dtype=np.uint8)
        parts += [cds[last:x], intron]
        last = x
    return np.concatenate(parts + [cds[last:]])


def _revcomp(x):
    return COMP[x[::-1]]


class _Query:
    def __init__(self, prot, nt, strand, score_only, profile=None):
        self.prot, self.nt, self.strand, self.score_only, self.profile = prot, nt, strand, score_only, profile


_blosum = None


def _profile(rng, prot):
    """Position-specific scores around the substitution matrix's rows, and gap costs that vary along the query."""
    global _blosum
    if _blosum is None:
        _blosum = mp.params_matrix(mp.mp_dp_default_params())
    out = np.zeros((len(prot) + 1, 23), dtype=np.int64)
    out[1:, :20] = _blosum[:20, :20].T[prot] + rng.integers(-1, 2, (len(prot), 20))
    out[1:, 20] = -23
    out[:, 21] = rng.integers(9, 14, len(prot) + 1)
    out[:, 22] = rng.integers(1, 3, len(prot) + 1)
    return out


def _pairs(mix, n, shape, seed, profile=False):
    rng = np.random.default_rng([shape, seed])
    out = []
    for g in _genes(np.random.default_rng(shape), mix, n):
        prot = _protein(rng, g[0])
        nt = GC40[rng.integers(0, 10, _nt_len(g))]
        if not g[6]:                                     # a score-only decoy has no gene in its region
            nt[g[2]:len(nt) - g[2]] = _spliced(rng, prot, g)
        if g[5] < 0:
            nt = _revcomp(nt)
        out.append(_Query(AA[prot].tobytes(), nt.tobytes(), g[5], g[6], _profile(rng, prot) if profile else None))
    return out


def _genome_with_regions(case, seed):
    rng = np.random.default_rng([case["shape"], seed])
    genes, at, spans, win = _region_sizes(case)
    genome = GC40[rng.integers(0, 10, case["genome"], dtype=np.uint8)]
    prots = []
    for g, x, s in zip(genes, at, spans):
        prot = _protein(rng, g[0])
        body = _spliced(rng, prot, g)[:s]
        genome[x:x + s] = body if g[5] > 0 else _revcomp(body)
        prots.append(AA[prot])
    return genome, prots, win


def _genome_with_proteome(case, seed):
    rng = np.random.default_rng([case["shape"], seed])
    lens, planted = _proteome(case)
    genome = GC40[rng.integers(0, 10, case["genome"], dtype=np.uint8)]
    off = np.concatenate([[0], np.cumsum(lens)])
    prot = _protein(rng, int(off[-1]))
    for k in range(planted):
        g = (int(lens[k]), [700, 1500], 0, 0.2, [], 1 if k % 2 else -1, False)
        body = _spliced(rng, prot[off[k]:off[k + 1]], g)
        x = int(rng.integers(0, max(1, case["genome"] - len(body))))
        body = body[:case["genome"] - x]
        genome[x:x + len(body)] = body if g[5] > 0 else _revcomp(body)
    return genome, AA[prot], off[:-1].astype(np.uint64), lens.astype(np.uint32)


# -------------------------------------------------------------- the calls
class State:
    """What the calling program holds: a context, and the batch, index or sequences it calls it with."""

    def __init__(self, case, **params):
        self.kind = case["kind"]
        self.ctx = mp.mp_dp_init(mp.mp_dp_default_params(**params), 0)
        self.batch = self.index = None

    def __del__(self):
        if self.batch is not None:
            mp.mp_dp_batch_free(self.ctx, self.batch)
        if self.index is not None:
            mp.mp_index_free(self.index)
        mp.mp_dp_destroy(self.ctx)


def _room(prot_lens):
    return sum(m + 16 for m in prot_lens)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "align":
        s = State(case, mode=case["mode"])
        queries = _pairs(case["mix"], case["n"], case["shape"], seed, case["profile"])
        s.pairs, s.room = mp.PairBatch(queries), _room(len(q.prot) for q in queries)
        if case["resident"]:
            s.batch = mp.mp_dp_batch_upload(s.ctx, s.pairs)
    elif kind == "regions":
        s = State(case, exon_rescore=1 if case["rescore"] else 0)
        genome, prots, win = _genome_with_regions(case, seed)
        lens = np.array([len(p) for p in prots])
        off = np.concatenate([[0], np.cumsum(lens)])
        who, at, size, strand = (np.array(c) for c in zip(*win))
        s.room = _room(lens[who].tolist())
        s.pairs = mp.RegionBatch(np.concatenate(prots), off[who], lens[who], genome, at, size, strand)
    elif kind == "serve":
        s = State(case)
        s.queries = [(q.prot, q.nt, q.strand) for q in _pairs("genes", case["n"], case["shape"], seed)]
        s.room = _room(len(q[0]) for q in s.queries)
    elif kind == "refine":
        s = State(case)
        s.pairs = mp.PairBatch(_pairs("genes", case["n"], case["shape"], seed))
    else:
        s = State(case)
        s.genome, s.prot, s.off, s.len = _genome_with_proteome(case, seed)
        if kind == "chain":
            s.index = mp.mp_index_build(s.ctx, s.genome)
    return s


def _cigars(ptr, n, room):
    """The CIGARs, one after the other, from where the library keeps them until its next call (zeros after the last:
    room, the residues and a few more per pair, is the same for every seed)."""
    has = n > 0
    ptr, n = ptr[has].astype(np.int64), n[has].astype(np.int64)
    out = np.zeros(room, dtype=np.uint32)
    if not len(n):
        return out
    if np.array_equal(ptr[1:], ptr[:-1] + 4 * n[:-1]):
        raw = ctypes.string_at(int(ptr[0]), int(4 * n.sum()))
    else:
        raw = b"".join(ctypes.string_at(p, 4 * k) for p, k in zip(ptr.tolist(), n.tolist()))
    out[:int(n.sum())] = np.frombuffer(raw, dtype=np.uint32)
    return out


def _results(r, room):
    out = {k: r[k] for k in ("score", "status", "prot_st", "prot_en", "nt_st", "nt_en", "n_cigar", "exon_score")}
    out["cigar"] = _cigars(r["cigar"], r["n_cigar"], room)
    return out


def _chains(ch, n):
    there = np.arange(ch.shape[1])[None, :] < n[:, None]
    return {"n_chains": n, **{k: np.where(there, ch[k], 0) for k in ch.dtype.names}}


TOP = 3


def run(s):
    if s.kind == "align" and s.batch is not None:
        mp.mp_dp_batch_run(s.ctx, s.batch)
        mp.mp_dp_batch_sync(s.ctx)
        return _results(mp.mp_dp_batch_download(s.ctx, s.batch, raw=True), s.room)
    if s.kind in ("align", "regions"):
        return _results(mp.mp_dp_align_batch(s.ctx, s.pairs, raw=True), s.room)
    if s.kind == "serve":
        tickets = [mp.mp_dp_submit(s.ctx, q) for q in s.queries]
        got = [mp.mp_dp_poll(s.ctx, t) for t in tickets]
        out = {k: np.array([g[k] for g in got]) for k in ("score", "status", "prot_st", "prot_en", "nt_st", "nt_en")}
        words = [w for g in got for w in g["cigar_raw"]]
        out["cigar"] = np.zeros(s.room, dtype=np.int64)
        out["cigar"][:len(words)] = words
        return out
    if s.kind == "refine":
        got = mp.mp_chain_refine(s.ctx, s.pairs)
        return {k: got[k] for k in got.dtype.names if k != "reserved"}
    if s.kind == "map":
        index = mp.mp_index_build(s.ctx, s.genome)
        out = _chains(*mp.mp_index_chain(s.ctx, index, s.prot, s.off, s.len, TOP))
        mp.mp_index_free(index)
        return out
    return _chains(*mp.mp_index_chain(s.ctx, s.index, s.prot, s.off, s.len, TOP))


# ------------------------------------------------------------------- work
# integer operations per cell of the recurrence: its 27 maxima and additions and one running maximum
CELL_OPS = 28


def work(case):
    """Sequences in, results out; for the aligner the recurrence's integer operations, for the second chaining round
    one comparison per protein 5-mer and base.  A protein 6-mer has about 20 entries in a 50 Mb index."""
    kind = case["kind"]
    if kind in ("align", "serve", "refine"):
        genes = _genes(np.random.default_rng(case["shape"]), case.get("mix", "genes"), case["n"])
        sizes = [(g[0], _nt_len(g)) for g in genes]
    elif kind == "regions":
        genes, _, _, win = _region_sizes(case)
        sizes = [(genes[w[0]][0], w[2]) for w in win]
        seqs = case["genome"] + sum(g[0] for g in genes)
    else:
        lens, _ = _proteome(case)
        hits = float(lens.sum()) * 20 * case["genome"] / 50e6
        out = case["n"] * (4 + 48 * TOP)
        return {"bytes": float(lens.sum()) + 4 * hits + out + (case["genome"] if kind == "map" else 0), "flops": 0.0}
    if kind != "regions":
        seqs = sum(m + n for m, n in sizes)
    cells = float(sum(m * n for m, n in sizes))
    if kind == "refine":
        return {"bytes": float(seqs + 48 * len(sizes)), "flops": float(sum(n for _, n in sizes))}
    return {"bytes": float(seqs + 32 * len(sizes)), "flops": CELL_OPS * cells}


# ------------------------------------------------------------------ exact
def _best_score(prot, nt, mat):
    """The best local score by the recurrence in 64 bits, one row of the genome at a time (default costs)."""
    q, e, f, r, stop = 11, 1, 23, 29, 23
    low = -(1 << 40)
    n, m = len(nt), len(prot)
    t = np.full(n + 8, 9)                                # t[x + 2] is base x (1-based); 9 outside
    t[3:n + 3] = np.searchsorted(ACGT, nt)
    b = lambda x: int(t[x + 2])  # noqa: E731

    def donor(x):
        k = (b(x + 1), b(x + 2))
        return {(2, 3): {0: 0, 2: 0, 1: 8, 3: 8}.get(b(x + 3), 30), (2, 1): 15, (0, 3): 21}.get(k, 30)

    def acceptor(x):
        k = (b(x - 1), b(x))
        return {(0, 2): {1: 0, 3: 0, 0: 8, 2: 8}.get(b(x - 2), 30), (0, 1): 21}.get(k, 30)

    order = AA.tobytes().decode()
    zero, none = np.zeros(m + 1, dtype=np.int64), np.full(m + 1, low, dtype=np.int64)
    H, D, A, B, C = [none, none, zero], [none] * 3, none, none, none
    d_before = donor(0)
    step = e * np.arange(m + 1)
    best = 0
    left = lambda v: np.concatenate([[low], v[:-1]])  # noqa: E731
    for i in range(1, n + 1):
        h1, h2, h3 = H[2], H[1], H[0]
        d0, d1 = donor(i), donor(i + 1)
        A = np.maximum(h1 - r - d_before, A)
        B = np.maximum(left(h1) - r - d0, B)
        C = np.maximum(left(h1) - r - d1, C)
        d_before = d0
        Dn = np.maximum(h3 - q - e, D[0] - e)
        h = np.maximum.reduce([zero, Dn, left(h1) - f, left(h2) - f, h1 - f, h2 - f, A - acceptor(i),
                               B - acceptor(i - 2), C - acceptor(i - 1)])
        if i >= 3:
            a = CODON_AA[b(i - 2) * 16 + b(i - 1) * 4 + b(i)]
            s = np.full(m, -stop) if a == "*" else mat[order.index(a)][prot]
            h[1:] = np.maximum(h[1:], h3[:-1] + s)
        h[0] = 0
        run_ = np.maximum.accumulate(h + step)           # I: the best opening to the left
        h[1:] = np.maximum(h[1:], run_[:-1] - q - step[1:])
        best = max(best, int(h.max()))
        H, D = [h2, h1, h], [D[1], D[2], Dn]
    return best


def exact(case, seed):
    """The best scores of small local batches; the other outputs follow from the library's tie rules."""
    if case["kind"] != "align" or case["mode"] != 0 or case["profile"] or case["n"] > 8 or case["mix"] != "one":
        return None
    mat = mp.params_matrix(mp.mp_dp_default_params()).astype(np.int64)
    out = {k: None for k in ("status", "prot_st", "prot_en", "nt_st", "nt_en", "n_cigar", "exon_score", "cigar")}
    score = []
    for p in _pairs(case["mix"], case["n"], case["shape"], seed):
        nt = np.frombuffer(p.nt, dtype=np.uint8)
        prot = np.searchsorted(np.sort(AA), np.frombuffer(p.prot, dtype=np.uint8))
        score.append(_best_score(np.argsort(AA)[prot], nt if p.strand > 0 else _revcomp(nt), mat))
    out["score"] = np.array(score)
    return out
