"""Counting plans and the sizes of a batch's sets: what a plan changes in the
unit counting does not keep a set from the super-k-mers that it takes by
default, and a plan tuned on a large set leaves the small ones their route."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _profile_of_count(mh, ctx, a, o, k):
    reads = mh.mh_pack_reads(ctx, a, o)
    ctx.profile_reset()
    g = mh.mh_count_kmers(ctx, reads, k, 2).numpy()
    return g, {name for name, (launches, _, _) in ctx.profile().items() if launches}


@pytest.mark.parametrize("k,n_reads", [(31, 3000), (31, 40_000), (61, 60_000)])
@pytest.mark.parametrize("delta", [-1, 0, 1])
def test_unit_bits_do_not_choose_the_route(k, n_reads, delta):
    import paper_1409_7208_gb300 as mh

    a, o = synth.uniform_genome_reads(5, 200_000, n_reads, 150, 0.01)
    ctx = mh.Context(device=0, profile=True)
    want, _ = _profile_of_count(mh, ctx, a, o, k)
    mh.mh_set_count_plan(ctx, path=0, sort_shape=0, unit_bits_delta=delta, spread_bits_delta=0, bucket_bits=-1)
    got, prof = _profile_of_count(mh, ctx, a, o, k)
    assert "super_count" in prof
    assert np.array_equal(got["keys"], want["keys"]) and np.array_equal(got["counts"], want["counts"])


def test_autotuned_batch_counts_its_small_sets_by_super_kmers():
    import paper_1409_7208_gb300 as mh

    # one set above 2^22 windows, the others below
    sets = [synth.uniform_genome_reads(80 + i, 300_000, n, 150, 0.01) for i, n in enumerate((50_000, 9000, 4000))]
    ctx = mh.Context(device=0, profile=True)
    mh.mh_run_batch(ctx, sets, 31, 2, workers=2, autotune=True)
    plan = mh.mh_get_count_plan(ctx)
    assert plan["path"] == 0 and plan["unit_bits_delta"] == 0, plan
    for a, o in sets:
        assert "super_count" in _profile_of_count(mh, ctx, a, o, 31)[1]
