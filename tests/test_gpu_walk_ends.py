"""Walks in graphs of short paths take no links, walks in one of long paths do;
the same contigs either way (MH_WALK_LINKS=1 and 0).  More than 2^22 edges, from
which on the dead ends are counted first."""
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
k, max_len = int(sys.argv[2]), int(sys.argv[3])
if sys.argv[1] == "short":
    a, o = synth.random_reads(k, 100_000, 150, 150)
else:
    a, o = synth.uniform_genome_reads(k, 2_500_000, 400_000, 150, 0.0)
ctx = mh.Context(device=0, profile=True)
s = mh.mh_count_kmers(ctx, mh.mh_pack_reads(ctx, a, o), k, 1)
assert s.view().n > 1 << 22
c = mh.mh_walk_contigs(ctx, s, None, 500, max_len, 3).numpy()
print(hashlib.sha256(c["ascii"].tobytes() + c["offs"].tobytes()).hexdigest(), "walk_links" in ctx.profile())
""" % ROOT


@pytest.mark.parametrize("paths,k,max_len", [("short", 31, 2000), ("short", 61, 2000), ("long", 31, 1000), ("long", 61, 2000)])
def test_links_by_dead_ends(paths, k, max_len):
    got = []
    for env in ({}, {"MH_WALK_LINKS": "1"}, {"MH_WALK_LINKS": "0"}):
        p = subprocess.run([sys.executable, "-c", CHILD, paths, str(k), str(max_len)], env=dict(os.environ, **env),
                           capture_output=True, text=True, timeout=600)
        assert p.returncode == 0, p.stdout + p.stderr
        got.append(p.stdout.split())
    assert got[0][0] == got[1][0] == got[2][0]
    assert [g[1] for g in got] == [str(paths == "long"), "True", "False"]
