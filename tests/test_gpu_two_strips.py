"""Warps that run one strip or two strips of a pair at once: results equal the
oracle's (whole numbers, no tolerance) at the edges of strips and chunks, with
an even and an odd number of strips, in every mode, for profile queries,
score-only pairs and every build of the kernel.  A batch of a few hundred
pairs runs one strip per warp (every pair's own chain of steps is longer than
a warp's share of the work), the same pairs many times over two."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

KEYS = ("score", "prot_st", "prot_en", "nt_st", "nt_en", "cigar")
# one strip; two; three (the first alone); four; five; a ragged and a full last strip
PROT = (64, 65, 127, 128, 129, 191, 192, 193, 255, 256, 257, 320)
# chunks of 96 steps; 63 and 127 steps after the last row; fewer rows than a codon
NT = (1, 2, 3, 31, 32, 33, 64, 65, 95, 96, 97, 129, 160, 161, 191, 192, 193, 225, 257, 321, 705)


@pytest.fixture(scope="module")
def mp():
    from paper_2210_08052_gb300 import build
    build.build()
    import paper_2210_08052_gb300 as m
    m.lib()
    return m


def _pairs(seed):
    rng = np.random.default_rng(seed)
    out = []
    for m in PROT:
        for n in NT:
            prot = synth.random_protein(rng, m)
            nt = synth.random_dna(rng, n)
            if rng.random() < 0.7:
                x = 3 * int(rng.integers(0, m))            # the region codes for a stretch of the protein
                nt = (synth.random_dna(rng, int(rng.integers(0, 20))) + synth.reverse_translate(rng, prot)[x:] +
                      nt)[:n]
            out.append(synth.Pair(prot, nt, 1 if rng.random() < 0.5 else -1))
    return out


# copies of the pairs: few pairs, one strip per warp; many, two
COPIES = pytest.mark.parametrize("copies", [1, 30])


def _params(mp, orc, mode, **more):
    p = mp.mp_dp_default_params(mode=mode, **more)
    op = orc.make_params(q=p.q, e=p.e, f=p.f, r=p.r, stop=p.stop, splice_model=p.splice_model, splice_p=p.splice_p)
    op.mode = mode
    return p, op


def _bad(pairs, got, want, keys=KEYS):
    return [(len(p.prot), len(p.nt), [k for k in keys if g[k] != w[k]], g["status"])
            for p, g, w in zip(pairs, got, want) if any(g[k] != w[k] for k in keys) or g["status"] & 0xF0]


@COPIES
@pytest.mark.parametrize("costs", [dict(), dict(q=0, e=1, f=0, r=8, stop=4, splice_model=1, splice_p=3)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_edges_match_oracle(mp, orc, mode, costs, copies):
    pairs = _pairs(200 + mode)
    params, op = _params(mp, orc, mode, **costs)
    want = [orc.align(p.prot, p.nt, p.strand, op) for p in pairs] * copies
    pairs = pairs * copies
    c = mp.mp_dp_init(params, 0)
    try:
        for variant in (1, 0):
            mp.mp_dp_set_tuning(c, dict(dp16_variant=variant, overlap_waves=1, item_order=variant))
            assert not (bad := _bad(pairs, mp.mp_dp_align_batch(c, pairs), want)), bad[:5]
        alone = [synth.Pair(p.prot, p.nt, p.strand, True) for p in pairs]
        got = mp.mp_dp_align_batch(c, alone)
        keys = ("score", "prot_en") if mode != 1 else ("score",)
        assert not (bad := _bad(alone, got, want, keys)), bad[:5]
    finally:
        mp.mp_dp_destroy(c)


@COPIES
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_stored_h_at_the_edges(mp, orc, mode, copies):
    """Every stored H, read through the traceback's view of the stream."""
    pairs = [p for p in _pairs(210 + mode) if len(p.prot) in (65, 128, 129, 192, 257) and len(p.nt) in (3, 65, 97, 161, 705)]
    params, op = _params(mp, orc, mode)
    c = mp.mp_dp_init(params, 0)
    try:
        b = mp.mp_dp_batch_upload(c, pairs * (10 * copies if copies > 1 else 1))
        mp.mp_dp_batch_run(c, b)
        mp.mp_dp_batch_sync(c)
        for k, p in enumerate(pairs):
            got = mp.mp_dp_debug_h(c, b, k, len(p.nt), len(p.prot))
            want = orc.fill_h(p.prot, p.nt, p.strand, op)
            assert np.array_equal(got, want), (len(p.prot), len(p.nt), np.argwhere(got != want)[:4].tolist())
        mp.mp_dp_batch_free(c, b)
    finally:
        mp.mp_dp_destroy(c)


@COPIES
@pytest.mark.parametrize("mode", [0, 2])
def test_profile_edges(mp, orc, mode, copies):
    rng = np.random.default_rng(220 + mode)
    pairs = [p for p in _pairs(220 + mode) if len(p.nt) in (2, 65, 161, 321, 705)]
    mat = mp.params_matrix(mp.mp_dp_default_params())
    order = "ARNDCQEGHILKMFPSTWYV"
    for p in pairs:
        m = len(p.prot)
        prof = np.zeros((m + 1, 23), dtype=np.int64)
        prof[1:, :20] = [mat[:20, order.index(x)] for x in p.prot] + rng.integers(-1, 2, (m, 20))
        prof[1:, 20] = -23
        prof[:, 21] = rng.integers(8, 15, m + 1)
        prof[:, 22] = rng.integers(1, 4, m + 1)
        p.profile = prof
    params, _ = _params(mp, orc, mode)
    want = [orc.align(p.prot, p.nt, p.strand, orc.make_params(mode=mode, prof=p.profile)) for p in pairs]
    want, pairs = want * 4 * copies, pairs * 4 * copies
    c = mp.mp_dp_init(params, 0)
    try:
        assert not (bad := _bad(pairs, mp.mp_dp_align_batch(c, pairs), want)), bad[:5]
    finally:
        mp.mp_dp_destroy(c)


@COPIES
def test_withheld_rows_time_out(mp, copies):
    """With boundary rows withheld, every pair of two strips or more gives
    up after the short poll limit and says so; the context stays usable."""
    pairs = [p for p in _pairs(230) if len(p.nt) == 705] * 20 * copies
    c = mp.mp_dp_init(mp.mp_dp_default_params(wait_limit=200, debug_flags=mp.MP_DEBUG_NO_PUBLISH), 0)
    try:
        for _ in range(2):
            for p, g in zip(pairs, mp.mp_dp_align_batch(c, pairs)):
                assert bool(g["status"] & mp.MP_ST_TIMEOUT) == (len(p.prot) > 64), len(p.prot)
    finally:
        mp.mp_dp_destroy(c)
