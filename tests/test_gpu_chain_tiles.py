"""Chaining in tiles of 32 anchors: chains equal the oracle's (whole numbers)
where the tiling and the 32-bit scores could go wrong: anchor counts around
multiples of 32, dense repeats (many equal scores, thousands of anchors that
follow one chain at a loss), every anchor on one strand, proteins past 32,000
residues (64-bit scores), and regions with anchor counts around the limit
between one warp and eight.  Also the index of genomes whose buckets hold
thousands of entries, tiny genomes, and regions around multiples of the second
round's tile of 4,096 bases."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FIELDS = ("strand", "n_anchors", "score", "x_first", "x_last", "y_first", "y_last")
REFINE_FIELDS = ("n_anchors", "score", "x_first", "x_last", "y_first", "y_last")


@pytest.fixture(scope="module")
def mp():
    from paper_2210_08052_gb300 import build
    build.build()
    import paper_2210_08052_gb300 as m
    m.lib()
    return m


def _genome(rng, prots, strand):
    parts = []
    for p in prots:
        gene = synth.reverse_translate(rng, p)
        parts += [synth.random_dna(rng, int(rng.integers(200, 3000)), 0.4), gene if strand(rng) else synth.revcomp(gene)]
    return "".join(parts) + synth.random_dna(rng, 2000, 0.4)


@pytest.mark.parametrize("case", ["mixed", "one strand", "repeats", "long protein"])
def test_chains_equal_the_oracles(mp, orc, case):
    rng = np.random.default_rng(300 + len(case))
    base = [synth.random_protein(rng, int(m)) for m in rng.integers(40, 400, 30)]
    strand = (lambda r: True) if case == "one strand" else (lambda r: r.random() < 0.5)
    queries = [p[:k] for p in base[:6] for k in (6, 7, 37, 38, 39, 40, len(p))] + base
    planted = base * 2
    if case == "repeats":
        unit = synth.random_protein(rng, 12)
        planted = [unit * 20, base[0], unit * 33, base[0], unit * 8] + base
        queries += [unit * n for n in (2, 3, 5, 8, 30, 60)]
    if case == "long protein":
        queries = ["".join(base) * 6, "".join(reversed(base)) * 7]
        queries = [(q * 4)[:m] for q, m in zip(queries, (32_000, 33_000))] + base[:3]
        assert len(queries[1]) == 33_000
    genome = _genome(rng, planted, strand)
    off = np.concatenate([[0], np.cumsum([len(q) for q in queries])])
    ctx = mp.mp_dp_init(None, 0)
    try:
        idx = mp.mp_index_build(ctx, genome)
        got = {top: mp.mp_index_chain(ctx, idx, "".join(queries), off[:-1], np.diff(off), top) for top in (1, 200)}
        mp.mp_index_free(idx)
    finally:
        mp.mp_dp_destroy(ctx)
    woff, wpos = orc.build_index(genome)
    most = 0
    for k, q in enumerate(queries):
        anc = orc.anchors(woff, wpos, q)
        most = max(most, len(anc))
        for top, (ch, n) in got.items():
            want, _ = orc.chain(anc, top)
            have = [{f: int(ch[k, t][f]) for f in FIELDS} for t in range(int(n[k]))]
            assert have == want, (k, len(q), len(anc), top)
    assert most > 300


def test_second_round_around_the_block_limit(mp, orc):
    """Regions with 1 to about 2,000 anchors, dense ones among them."""
    rng = np.random.default_rng(320)
    pairs, counts = [], []
    for copies in (0, 1, 2, 3, 4, 5, 6, 8, 12):
        for m in (5, 6, 36, 37, 100, 170, 400):
            prot = synth.random_protein(rng, m)
            nt = synth.random_dna(rng, 400, 0.4) + "".join(
                synth.reverse_translate(rng, prot) + synth.random_dna(rng, int(rng.integers(0, 300)), 0.4)
                for _ in range(copies))
            strand = 1 if rng.random() < 0.5 else -1
            pairs.append(synth.Pair(prot, nt if strand > 0 else synth.revcomp(nt), strand))
    unit = synth.random_protein(rng, 9)
    for n in (3, 6, 9, 12):
        pairs.append(synth.Pair(unit * n, synth.reverse_translate(rng, unit * n), 1))
    ctx = mp.mp_dp_init(None, 0)
    try:
        got = mp.mp_chain_refine(ctx, pairs)
    finally:
        mp.mp_dp_destroy(ctx)
    for k, p in enumerate(pairs):
        anc = orc.refine_anchors(p.prot, p.nt, p.strand)
        counts.append(len(anc))
        want, _ = orc.refine_chain(anc)
        assert {f: int(got[k][f]) for f in REFINE_FIELDS} == want, (k, len(anc))
    assert any(c > 512 for c in counts) and any(0 < c <= 512 for c in counts) and any(c == 0 for c in counts)


@pytest.mark.parametrize("case", ["repeats", "tiny"])
def test_index_of_full_buckets_and_tiny_genomes(mp, orc, case):
    rng = np.random.default_rng(330)
    unit = synth.reverse_translate(rng, synth.random_protein(rng, 40))
    genomes = [synth.random_dna(rng, 700, 0.4) + unit * 900 + synth.revcomp(unit) * 300 + "N" + unit * 41]
    if case == "tiny":
        gene = synth.reverse_translate(rng, synth.random_protein(rng, 400))
        genomes = [gene[:n] for n in (0, 1, 2, 3, 90, 107, 108, 109, 255, 256, 257, 511, 512, 513, 1200)]
        genomes.append(synth.random_dna(rng, 3 * 1024 * 3 + 1, 0.4) + gene)
    ctx = mp.mp_dp_init(None, 0)
    try:
        for g in genomes:
            idx = mp.mp_index_build(ctx, g)
            off, ent = mp.mp_index_download(ctx, idx)
            prot = synth.random_protein(rng, 5) + "MKVLAWDERT" * 3
            ch, n = mp.mp_index_chain(ctx, idx, prot, [0], [len(prot)], 5)
            mp.mp_index_free(idx)
            woff, went = orc.build_index(g)
            assert (off == woff).all() and (ent == went).all(), len(g)
            want, _ = orc.chain(orc.anchors(woff, went, prot), 5)
            assert [{f: int(ch[0, t][f]) for f in FIELDS} for t in range(int(n[0]))] == want
        if case == "repeats":
            assert np.diff(off.astype(np.int64)).max() > 512
    finally:
        mp.mp_dp_destroy(ctx)


def test_second_round_around_the_tiles(mp, orc):
    rng = np.random.default_rng(340)
    pairs = []
    for L in (14, 15, 16, 4109, 4110, 4111, 4112, 8205, 8206, 8207, 12302):
        for strand in (1, -1):
            prot = synth.random_protein(rng, int(rng.integers(6, 300)))
            nt = synth.random_dna(rng, L, 0.4)
            gene = synth.reverse_translate(rng, prot)
            for at in (0, 4096 - 40, 4096 + 8, 8192 - 100):
                nt = (nt[:at] + gene + nt[at + len(gene):])[:L]
            if L > 4096:
                nt = nt[:4093] + "N" + nt[4094:]
            pairs.append(synth.Pair(prot, nt if strand > 0 else synth.revcomp(nt), strand))
    ctx = mp.mp_dp_init(None, 0)
    try:
        got = mp.mp_chain_refine(ctx, pairs)
    finally:
        mp.mp_dp_destroy(ctx)
    for k, p in enumerate(pairs):
        want = orc.refine(p.prot, p.nt, p.strand)
        assert {f: int(got[k][f]) for f in REFINE_FIELDS} == want, (k, len(p.nt), p.strand)


def test_second_round_of_more_bytes_than_are_sent_at_once(mp):
    """Sequences go to the device in windows of 256 MB: the pairs of every
    window, the ones at its edges included, have the chains they have alone."""
    rng = np.random.default_rng(350)
    kinds = []
    for L in (7_000_000, 6_999_999, 5_000_003):
        prot = synth.random_protein(rng, 90)
        nt = synth.random_dna(rng, L - 270, 0.4)
        kinds.append(synth.Pair(prot, nt[:L // 2] + synth.reverse_translate(rng, prot) + nt[L // 2:], 1))
    pairs = [kinds[k % 3] for k in range(90)]
    assert sum(len(p.nt) + len(p.prot) for p in pairs) > 2 * (256 << 20)
    ctx = mp.mp_dp_init(None, 0)
    try:
        alone = [mp.mp_chain_refine(ctx, [p])[0] for p in kinds]
        got = mp.mp_chain_refine(ctx, pairs)
    finally:
        mp.mp_dp_destroy(ctx)
    for k in range(len(pairs)):
        assert all(int(got[k][f]) == int(alone[k % 3][f]) for f in REFINE_FIELDS), k
    # (the planted gene scores its length; of the links of equal worth along its
    # diagonal the one from the earliest anchor is taken, so its anchors are fewer)
    assert all(int(a["score"]) >= 90 << 16 for a in alone)
