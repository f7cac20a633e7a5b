"""The second chaining round of a region longer than the window (256 MB) in
which sequences go to the device: a gene across the window's edge is chained as
the oracle chains its surroundings, and so is the pair behind the region."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FIELDS = ("n_anchors", "score", "x_first", "x_last", "y_first", "y_last")
WINDOW = 256 << 20


def test_region_longer_than_a_window(orc):
    from paper_2210_08052_gb300 import build
    build.build()
    import paper_2210_08052_gb300 as mp

    rng = np.random.default_rng(360)
    prots = [synth.random_protein(rng, m) for m in (400, 90)]
    genes = [synth.reverse_translate(rng, p).encode() for p in prots]
    nt = np.frombuffer(b"ACGT", dtype=np.uint8)[rng.integers(0, 4, WINDOW + 20_000_000, dtype=np.uint8)]
    at = WINDOW - len(prots[0]) - 600                    # (the protein is sent before its region)
    nt[at:at + len(genes[0])] = np.frombuffer(genes[0], dtype=np.uint8)
    near, flank = nt[at - 20_000:at + 20_000].tobytes(), synth.random_dna(rng, 700).encode()
    pairs = [(prots[0].encode(), nt.tobytes(), 1, 0), (prots[1].encode(), flank + genes[1] + flank, 1, 0)]
    ctx = mp.mp_dp_init(None, 0)
    try:
        got = mp.mp_chain_refine(ctx, pairs)
    finally:
        mp.mp_dp_destroy(ctx)
    for k, (region, shift) in enumerate(((near, at - 20_000), (pairs[1][1], 0))):
        want = dict(orc.refine(prots[k], region.decode(), 1))
        want["x_first"] += shift
        want["x_last"] += shift
        assert {f: int(got[k][f]) for f in FIELDS} == want, k
