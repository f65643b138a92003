"""Counting by super-k-mers, forced on inputs small enough for the oracle by a
child process with MH_SUPER=1: every key width and minimizer length (k = 20,
24, 25, 30, 31, 32, 62, 63, 64, 127), d = 1 and 2, ragged reads with invalid
bytes, reads around tile ends, reads of one symbol thousands of bases long
(runs cut at tile ends), a read repeated 7,000 times, palindromes; bins that
fall to the unit counting (MH_SUPER_HOT: bins of more windows than that;
MH_SUPER_PROBES: keys that find no slot), some or all of them.  At sizes
where the route is the default, its tables equal the unit route's
(MH_SUPER=0), with and without the sampled sizing of the outputs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SMALL = r"""
import sys, numpy as np
sys.path.insert(0, %r)
import oracle, synth, paper_1409_7208_gb300 as mh
ctx = mh.Context(device=0, profile=True)
rng = np.random.default_rng(3)

def repeated():
    a, o = synth.uniform_genome_reads(5, 4000, 300, 150, 0.01)
    rep = bytes(a[:140])
    return synth.reads_from_strings([rep] * 7000 + [bytes(a[int(o[i]):int(o[i + 1])]) for i in range(len(o) - 1)])

def odd():
    g = "".join("ACGT"[i] for i in rng.integers(0, 4, 5000))
    rc = lambda s: s[::-1].translate(str.maketrans("ACGT", "TGCA"))
    pal = [g[i:i + 70] + rc(g[i:i + 70]) for i in range(0, 2000, 97)]
    return synth.reads_from_strings(["A" * 5000, "T" * 2047, "C" * 2048, "ACGT" * 600, "AC" * 900, "", g, g, rc(g), "N" * 50,
                                     g[:2049], "G" * 30 + "N" + "G" * 200] + pal + pal + [g[i:i + 131] for i in range(300)])

sets = {"genome": synth.uniform_genome_reads(1, 4000, 2000, 150, 0.01), "ragged": synth.random_reads(6, 600, 0, 300, p_invalid=0.01),
        "repeated": repeated(), "odd": odd()}
for name, (a, o) in sets.items():
    for k in [int(x) for x in sys.argv[1].split(",")]:
        for d in (1, 2):
            reads = mh.mh_pack_reads(ctx, a, o)
            s = mh.mh_count_kmers(ctx, reads, k, d)
            m = mh.mh_mercy_kmers(ctx, reads, s)
            w = oracle.count(a, o, k, d, mercy=True)
            gs, gm = s.numpy(), m.numpy()
            for got, want in ((gs["keys"], w["solid_keys"]), (gs["counts"], w["solid_cnt"]),
                              (gm["keys"], w["mercy_keys"]), (gm["counts"], w["mercy_cnt"])):
                assert np.array_equal(got, want), (name, k, d)
            assert gs["n_kmers"] == w["n_kmers"] and gs["n_distinct"] == w["n_distinct"], (name, k, d)
prof = ctx.profile()
assert "super_count" in prof
assert "super_expand" in prof or sys.argv[2] != "rest", sorted(prof)
print("ok")
""" % ROOT


def _child(code, args, env):
    p = subprocess.run([sys.executable, "-c", code] + args, env=dict(os.environ, **env), capture_output=True, text=True,
                       timeout=900)
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout


@pytest.mark.parametrize("ks", ["20,24", "25,30,31", "32,62,63", "64,127"])
@pytest.mark.parametrize("env", [{"MH_SUPER_HOT": str(1 << 30)}, {"MH_SUPER_HOT": "0"}, {"MH_SUPER_HOT": "1500", "MH_SUPER_PROBES": "1"}],
                         ids=["bins", "all_rest", "some_rest"])
def test_small_sets_match_oracle(ks, env):
    assert "ok" in _child(SMALL, [ks, "bins" if env["MH_SUPER_HOT"] == str(1 << 30) else "rest"], dict(env, MH_SUPER="1"))


LARGE = r"""
import sys, hashlib, numpy as np
sys.path.insert(0, %r)
import synth, paper_1409_7208_gb300 as mh
k, pairs, sigma = int(sys.argv[1]), int(sys.argv[2]), float(sys.argv[3])
ctx = mh.Context(device=0, profile=True)
a, o = synth.metagenome_reads(seed=4, n_genomes=5, median_len=3e5, sigma_ab=sigma, n_pairs=pairs)
reads = mh.mh_pack_reads(ctx, a, o)
s = mh.mh_count_kmers(ctx, reads, k, 2)
m = mh.mh_mercy_kmers(ctx, reads, s)
v = s.view()
h = hashlib.sha256()
for x in (s.numpy(), m.numpy()):
    h.update(x["keys"].tobytes()); h.update(x["counts"].tobytes())
print(h.hexdigest(), v.n, v.n_kmers, v.n_distinct, "super_count" in ctx.profile())
""" % ROOT


@pytest.mark.parametrize("k,pairs,sigma", [(31, 18_000, 1.0), (31, 150_000, 1.5), (21, 150_000, 1.5), (47, 200_000, 1.5),
                                           (99, 400_000, 2.0)])
def test_equals_unit_route(k, pairs, sigma):
    new = _child(LARGE, [str(k), str(pairs), str(sigma)], {}).split()
    old = _child(LARGE, [str(k), str(pairs), str(sigma)], {"MH_SUPER": "0"}).split()
    assert new[:-1] == old[:-1]
    assert (new[-1], old[-1]) == ("True", "False")
