"""A graph built of two tables that share edges (mh_build_sdbg accepts any two
of one k): each shared edge is an entry of its own, so a group of entries holds
up to 32 of them, and the nodes and the padding are those of the union.  Groups
of 26 entries, some of them across the tiles of the zero-degree join (2,048,
1,024 and 512 entries for 1, 2 and 4 key words), where the last edge alone has
its target."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [21, 40, 80])
@pytest.mark.parametrize("first", [0, 6])
def test_a_table_built_with_itself(k, first):
    import paper_1409_7208_gb300 as mh

    rng = np.random.default_rng(k)
    ends = [(a, b) for a in range(4) for b in range(3)] + [(3, 3)]
    # (the smallest core shifts the groups behind it)
    reads = ["ACGT"[a] + "A" * (k - 1) + "ACGT"[b] for a, b in ends[:first]]
    for _ in range(300):
        core = "".join("ACGT"[i] for i in rng.integers(0, 4, k - 1))
        reads += ["ACGT"[a] + core + "ACGT"[b] for a, b in ends]
    ascii, offs = synth.reads_from_strings(reads)
    ctx = mh.Context(device=0)
    solid = mh.mh_count_kmers(ctx, mh.mh_pack_reads(ctx, ascii, offs), k, 1)
    one, two = mh.mh_build_sdbg(ctx, solid, None).numpy(), mh.mh_build_sdbg(ctx, solid, solid).numpy()
    for f in ("t", "u", "n_nodes"):
        assert two[f] == one[f], f
    assert np.array_equal(two["aux"], one["aux"])
    # an edge's second entry follows its first and has the minus flag
    n = solid.view().n
    assert two["m"] == one["m"] + n
    assert np.count_nonzero(two["W"] > 4) == np.count_nonzero(one["W"] > 4) + n
