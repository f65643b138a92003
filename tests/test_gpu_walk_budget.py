"""A walk under a budget with room for the links of its edges but not for
the finer index that making them takes: it walks by search instead, with the
same contigs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [21, 47])
def test_links_that_do_not_fit_are_left_out(k):
    import paper_1409_7208_gb300 as mh

    a, o = synth.uniform_genome_reads(k, 400_000, 60_000, 150, 0.01)

    def walk(ctx, solid):
        c = mh.mh_walk_contigs(ctx, solid, None, 100, 2000, 5)
        g = c.numpy()
        c.free()
        return g["ascii"].tobytes(), g["offs"].tobytes()

    plain = mh.Context(device=0)
    solid = mh.mh_count_kmers(plain, mh.mh_pack_reads(plain, a, o), k, 2)
    want = walk(plain, solid)
    # between the links' 40 bytes an edge and what the call takes with them:
    # every budget that walked by search still walks
    n = solid.view().n
    for extra in np.linspace(0, 6 * n + 400_000, 9).astype(int):
        ctx = mh.Context(device=0, hbm_budget=40 * n + 100 * (2000 // 4 + 64) + int(extra), profile=True)
        assert walk(ctx, solid) == want
        ctx.close()
