"""A protein or pair with 2^31 anchors or more is refused once its anchors are
counted, before any is written: predecessors are 32-bit and signed.  One of
fewer, of the same repeats, is chained."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    from paper_2210_08052_gb300 import build
    build.build()
    import paper_2210_08052_gb300 as m
    m.lib()
    return m


def _refused(mp, call):
    with pytest.raises(mp.MPError) as e:
        call()
    assert e.value.code == mp.MP_ETOOLARGE


def test_first_round(mp, orc):
    ctx = mp.mp_dp_init(None, 0)
    try:
        # poly-T: every frame of strand 0 reads F, whose 6-mer is sampled
        genome = "T" * 300_000
        idx = mp.mp_index_build(ctx, genome)
        prot = "F" * 8000
        off, ent = mp.mp_index_download(ctx, idx)
        assert len(ent) * (len(prot) - 5) >= 1 << 31
        _refused(mp, lambda: mp.mp_index_chain(ctx, idx, prot, [0], [len(prot)], 1))
        mp.mp_index_free(idx)
        genome = "T" * 1200
        idx = mp.mp_index_build(ctx, genome)
        prot = "F" * 9
        ch, n = mp.mp_index_chain(ctx, idx, prot, [0], [len(prot)], 3)
        mp.mp_index_free(idx)
        want, _ = orc.chain(orc.anchors(*orc.build_index(genome), prot), 3)
        assert int(n[0]) == len(want) > 0
        assert [{f: int(ch[0, t][f]) for f in want[0]} for t in range(len(want))] == want
    finally:
        mp.mp_dp_destroy(ctx)


def test_second_round(mp, orc):
    ctx = mp.mp_dp_init(None, 0)
    try:
        small = ("F" * 9, "T" * 200, 1, 0)
        large = ("F" * 8192, "T" * 300_000, 1, 0)
        assert 8188 * (300_000 - 14) >= 1 << 31
        _refused(mp, lambda: mp.mp_chain_refine(ctx, [small, large]))
        got = mp.mp_chain_refine(ctx, [small])[0]
        want = orc.refine(small[0], small[1], 1)
        assert {f: int(got[f]) for f in want} == want
    finally:
        mp.mp_dp_destroy(ctx)
