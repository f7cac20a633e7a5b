"""Which form the packed int16 kernel runs a pair in: one strip of 64 residues
per warp, or two.  Both give the same results, so the tests tell them apart by
the bytes that mp_dp_stats counts: a warp of two strips reads its pair's records
once for both (with 64 more steps), and hands boundary rows on half as often."""
import pytest

from test_gpu_two_strips import _pairs

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
