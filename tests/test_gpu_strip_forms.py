"""Which form the packed int16 kernel runs a pair in: one strip of 64 residues
per warp, or two.  Both give the same results, so the tests tell them apart by
the bytes that mp_dp_stats counts: a warp of two strips reads its pair's records
once for both (with 64 more steps), and hands boundary rows on half as often."""
import numpy as np
import pytest

import synth
from test_gpu_two_strips import _bad, _pairs, _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    from paper_2210_08052_gb300 import build
    build.build()
    import paper_2210_08052_gb300 as m
    m.lib()
    return m


def _counted(pairs, duo):
    """(record_read_bytes, boundary_bytes) of pairs run in one form."""
    read = rows = 0
    for p in pairs:
        n = len(p.nt)
        strips, chunks, chunks2 = -(-len(p.prot) // 64), -(-(n + 63) // 96), -(-(n + 127) // 96)
        twos = strips // 2 if duo else 0
        items = strips - twos
        read += ((items - twos) * (chunks + 1) + twos * (chunks2 + 1)) * 96 * 16
        rows += (items - 1) * chunks * 96 * 4
    return read, rows


@pytest.mark.parametrize("duo", [False, True])
def test_counters_follow_the_form(mp, duo):
    """A handful of pairs run one strip per warp; thousands, two."""
    pairs = [p for p in _pairs(240) if len(p.nt) in (65, 97, 705)]
    pairs = pairs * 200 if duo else [p for p in pairs if len(p.nt) == 705]
    c = mp.mp_dp_init(None, 0)
    try:
        mp.mp_dp_align_batch(c, pairs, raw=True)
        st = mp.mp_dp_get_stats(c)
    finally:
        mp.mp_dp_destroy(c)
    assert (st["record_read_bytes"], st["boundary_bytes"]) == _counted(pairs, duo)


def _copies(mp, c, pairs):
    """How many copies of the pairs make a warp's share of the steps (12 warps
    per SM) longer than every pair's own chain of steps, by half."""
    items = [-(-len(p.prot) // 128) for p in pairs]
    chain = max(len(p.nt) + 128 + 288 * (k - 1) for p, k in zip(pairs, items))
    steps = sum(k * (len(p.nt) + 127) for p, k in zip(pairs, items))
    return -(-3 * chain * mp.mp_dp_num_sms(c) * 12 // (2 * steps))


def _run(mp, c, pairs, duo):
    """Results of the pairs: all in one batch of two strips per warp, many times
    over, or in batches of at most a strip per SM (whose share is below the
    shortest chain), one strip per warp.  Returns (copies, results)."""
    copies = _copies(mp, c, pairs) if duo else 1
    batches = [pairs * copies] if duo else [[]]
    strips = 0
    for p in [] if duo else pairs:
        s = -(-len(p.prot) // 64)
        if strips + s > mp.mp_dp_num_sms(c):
            batches.append([])
            strips = 0
        batches[-1].append(p)
        strips += s
    got = []
    for batch in batches:
        got += mp.mp_dp_align_batch(c, batch)
        st = mp.mp_dp_get_stats(c)
        assert (st["record_read_bytes"], st["boundary_bytes"]) == _counted(batch, duo)
    return copies, got


FORM = pytest.mark.parametrize("duo", [False, True], ids=["one strip", "two strips"])


@FORM
@pytest.mark.parametrize("costs", [dict(), dict(q=0, e=1, f=0, r=8, stop=4, splice_model=1, splice_p=3)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_each_form_matches_the_oracle(mp, orc, mode, costs, duo):
    """Every edge of strips and chunks in the form that the batch is meant to
    run: alignments, and score-only pairs (global mode keeps its tracebacks)."""
    pairs = _pairs(250 + mode)
    params, op = _params(mp, orc, mode, **costs)
    want = [orc.align(p.prot, p.nt, p.strand, op) for p in pairs]
    c = mp.mp_dp_init(params, 0)
    try:
        n, got = _run(mp, c, pairs, duo)
        assert not (bad := _bad(pairs * n, got, want * n)), bad[:5]
        alone = [synth.Pair(p.prot, p.nt, p.strand, True) for p in pairs]
        n, got = _run(mp, c, alone, duo)
        keys = ("score", "prot_en") if mode != 1 else ("score",)
        assert not (bad := _bad(alone * n, got, want * n, keys)), bad[:5]
    finally:
        mp.mp_dp_destroy(c)


@FORM
@pytest.mark.parametrize("mode", [0, 2])
def test_each_form_of_profile_queries(mp, orc, mode, duo):
    rng = np.random.default_rng(260 + mode)
    pairs = [p for p in _pairs(260 + mode) if len(p.nt) in (2, 65, 161, 321, 705)]
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
    c = mp.mp_dp_init(params, 0)
    try:
        n, got = _run(mp, c, pairs, duo)
        assert not (bad := _bad(pairs * n, got, want * n)), bad[:5]
    finally:
        mp.mp_dp_destroy(c)


def test_poll_limit_bounds_both_kernels_waits_alike(mp):
    """With boundary rows withheld, a pair of three strips waits out its poll
    limit, at most a fifth of a second, and is marked.  The int16 wait lasts as
    long as the int32 kernel's under the same limit (less 5 per cent: a poll's load
    may take a little less)."""
    rng = np.random.default_rng(270)
    pair = synth.Pair(synth.random_protein(rng, 192), synth.random_dna(rng, 300), 1)
    ms = []
    for force_int32 in (0, 1):
        c = mp.mp_dp_init(mp.mp_dp_default_params(wait_limit=40_000, debug_flags=mp.MP_DEBUG_NO_PUBLISH,
                                                  force_int32=force_int32), 0)
        try:
            mp.mp_dp_set_timing(c, True)
            for _ in range(3):
                assert mp.mp_dp_align_batch(c, [pair])[0]["status"] & mp.MP_ST_TIMEOUT
            ms.append(mp.mp_dp_get_stats(c)["dp_ms"])
        finally:
            mp.mp_dp_destroy(c)
    assert ms[0] > 0.95 * ms[1], ms
