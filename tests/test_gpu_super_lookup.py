"""Lookups of windows in the super-k-mer bins by the mercy step: the same
edges as by the ascending spectrum (MH_SUPER=0), for every key width, and not
much slower; thin coverage, so that gaps and lookups are many."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, %r)
import hashlib
import synth, paper_1409_7208_gb300 as mh
k, n_reads = int(sys.argv[1]), int(sys.argv[2])
a, o = synth.uniform_genome_reads(k, 30 * n_reads, n_reads, 150, 0.02)
ctx = mh.Context(device=0, profile=True)
reads = mh.mh_pack_reads(ctx, a, o)
s = mh.mh_count_kmers(ctx, reads, k, 2)
best = 1e9
for _ in range(4):
    ctx.profile_reset()
    m = mh.mh_mercy_kmers(ctx, reads, s)
    p = ctx.profile()
    best = min(best, sum(p[x][1] for x in ("mercy_walk", "mercy_spectrum_index") if x in p))
g = m.numpy()
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), len(g["counts"]), "super_count" in ctx.profile(), best)
""" % ROOT


def _run(k, n_reads, env):
    p = subprocess.run([sys.executable, "-c", CHILD, str(k), str(n_reads)], env=dict(os.environ, **env), capture_output=True,
                       text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout.split()


@pytest.mark.parametrize("k", [31, 33, 47, 61, 64, 99, 127])
def test_lookups_in_bins(k):
    bins, index = _run(k, 600_000, {}), _run(k, 600_000, {"MH_SUPER": "0"})
    assert bins[:2] == index[:2] and int(bins[1]) > 0 and (bins[2], index[2]) == ("True", "False")
    # a window's minimizer besides, an index to build less
    assert float(bins[3]) <= 1.4 * float(index[3]), (bins, index)
