"""Tile edges of the graph's emission (2,048 final positions a CTA) and of the
mercy step's grouped lookups (four windows a group, up to 32 fragments a warp),
against the oracle: whole numbers, so every array is equal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _dna(rng, n):
    return "".join("ACGT"[i] for i in rng.integers(0, 4, n))


def _check(ascii, offs, k, d, with_mult=False):
    import paper_1409_7208_gb300 as mh

    ctx = mh.Context(device=0, with_mult=with_mult)
    reads = mh.mh_pack_reads(ctx, ascii, offs)
    solid = mh.mh_count_kmers(ctx, reads, k, d)
    mercy = mh.mh_mercy_kmers(ctx, reads, solid)
    got_g, got_s, got_m = mh.mh_build_sdbg(ctx, solid, mercy).numpy(), solid.numpy(), mercy.numpy()
    w = oracle.count(ascii, offs, k, d, mercy=True)
    g = oracle.build_sdbg(k, w["solid_keys"], w["solid_cnt"], w["mercy_keys"], w["mercy_cnt"])
    assert np.array_equal(got_s["keys"], w["solid_keys"]) and np.array_equal(got_s["counts"], w["solid_cnt"])
    assert np.array_equal(got_m["keys"], w["mercy_keys"]) and np.array_equal(got_m["counts"], w["mercy_cnt"])
    for f in ("W", "last", "valid", "dummy", "aux", "F"):
        assert np.array_equal(np.asarray(got_g[f]), np.asarray(g[f])), f
    if with_mult:
        assert np.array_equal(got_g["mult"], g["mult"])
    return got_g["m"], len(got_m["counts"])


@pytest.mark.parametrize("k", [21, 40, 80])
@pytest.mark.parametrize("m", [6, 2046, 2048, 2050, 6144, 8194])
def test_emission_around_tiles(k, m):
    # one read: two chains of m / 2 - 2 edges, each with a dummy and a $ entry
    a, o = synth.reads_from_strings([_dna(np.random.default_rng(m + k), (m - 4) // 2 + k)])
    assert _check(a, o, k, 1)[0] == m


@pytest.mark.parametrize("k,n", [(21, 341), (21, 342), (33, 1500), (70, 700)])
def test_emission_mostly_padding(k, n):
    # reads of one window: two edges, two dummies and two $ entries each
    rng = np.random.default_rng(n)
    a, o = synth.reads_from_strings([_dna(rng, k + 1) for _ in range(n)])
    assert _check(a, o, k, 1)[0] == 6 * n


@pytest.mark.parametrize("k", [4, 12, 21, 31, 32, 47, 63, 64, 99])
@pytest.mark.parametrize("n", [37, 3000])
def test_mercy_groups(k, n):
    # thin coverage of one genome by reads of 0 to 9 windows and a few long
    # ones, some of them with a gap's worth of errors or an N
    rng = np.random.default_rng(k * n)
    g = _dna(rng, 40 + k + n // 2)
    reads = []
    for i in range(n):
        ln = int(rng.integers(k, k + 10)) if i % 5 else int(rng.integers(k, 3 * k + 60))
        s = int(rng.integers(0, max(1, len(g) - ln)))
        r = list(g[s:s + ln])
        if i % 3 == 0:
            r[int(rng.integers(0, len(r)))] = "ACGTN"[int(rng.integers(0, 5))]
        reads.append("".join(r))
    a, o = synth.reads_from_strings(reads)
    _check(a, o, k, 2, with_mult=True)


@pytest.mark.parametrize("k,n", [(21, 1), (21, 16), (21, 8191), (21, 8192), (21, 8193), (40, 4095), (40, 4097), (80, 2048), (80, 2049)])
def test_sorts_around_one_cta(k, n):
    # 2 n dummies, sorted by one CTA up to 16,384 words of keys
    rng = np.random.default_rng(n)
    a, o = synth.reads_from_strings([_dna(rng, k + 1) for _ in range(n)])
    assert _check(a, o, k, 1)[0] == 6 * n


@pytest.mark.parametrize("where", ["inside", "edges", "empty_reads", "one_base_reads", "all_invalid", "long"])
def test_pack_around_tiles(where):
    # the compacting path works in tiles of 4,096 input bases, chunks of 16
    import paper_1409_7208_gb300 as mh

    rng = np.random.default_rng(9)
    if where == "inside":
        a, o = synth.random_reads(21, 2000, 0, 90, p_invalid=0.1)
    elif where == "edges":
        # reads and Ns at and beside the tiles' and chunks' ends
        g = list(_dna(rng, 5 * 4096 + 7))
        for p in (0, 15, 16, 31, 4095, 4096, 8190, 8191, 12287, 12289, 16384, len(g) - 1):
            g[p] = "N"
        g = "".join(g)
        a, o = synth.reads_from_strings([g[:4096], g[4096:8191], g[8191:8193], g[8193:12288], g[12288:]])
    elif where == "empty_reads":
        a, o = synth.reads_from_strings([""] * 300 + [_dna(rng, 4096), ""] + [""] * 700 + [_dna(rng, 4095), "", "A", "", _dna(rng, 33)] + [""] * 5)
    elif where == "one_base_reads":
        a, o = synth.reads_from_strings(["ACGTN"[i] for i in rng.integers(0, 5, 9000)])
    elif where == "all_invalid":
        a, o = synth.reads_from_strings(["N" * 5000, "", "nnn."])
    else:
        g = _dna(rng, 30_000)
        a, o = synth.reads_from_strings([g[:17_000] + "N" + g[17_000:]])
    bases, fo, fr = oracle.fragments(a, o)
    r = mh.mh_pack_reads(mh.Context(device=0), a, o).tensors()
    assert (r["n_frags"], r["n_packed"]) == (len(fr), len(bases))
    code = np.zeros(-(-len(bases) // 16) * 16, dtype=np.uint32)
    code[:len(bases)] = np.searchsorted(np.frombuffer(b"ACGT", np.uint8), np.frombuffer(bytes(bases), np.uint8))
    want = (code.reshape(-1, 16) << (30 - 2 * np.arange(16, dtype=np.uint32))).sum(axis=1, dtype=np.uint32)
    assert np.array_equal(r["packed"].cpu().numpy().view(np.uint32)[:len(want)], want)
    assert np.array_equal(r["frag_offs"].cpu().numpy().view(np.uint64), fo)
    assert np.array_equal(r["frag_read"].cpu().numpy().view(np.uint32), fr)
