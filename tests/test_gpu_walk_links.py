"""Contig walks by links and jumps (MH_WALK_LINKS=1) give the walks of the
search at every step (=0): walks that end at dead ends, at max_len within a
jump, and at k + 1; graphs with branches, of every key width, with and
without mercy edges."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, hashlib
sys.path.insert(0, %r)
import synth, paper_1409_7208_gb300 as mh
ctx = mh.Context(device=0)
h = hashlib.sha256()
for k, cover, lens in ((12, 30, (13, 300)), (31, 30, (32, 47, 48, 49, 2000)), (47, 8, (3000,)), (99, 4, (100, 103, 119, 4000))):
    a, o = synth.uniform_genome_reads(k, 30_000, cover * 200, 150, 0.01)
    reads = mh.mh_pack_reads(ctx, a, o)
    solid = mh.mh_count_kmers(ctx, reads, k, 2)
    for mercy in (mh.mh_mercy_kmers(ctx, reads, solid), None):
        for n in lens:
            c = mh.mh_walk_contigs(ctx, solid, mercy, 777, n, 5).numpy()
            h.update(c["ascii"].tobytes()); h.update(c["offs"].tobytes())
print(h.hexdigest())
""" % ROOT


def test_links_give_the_same_walks():
    got = []
    for v in ("1", "0"):
        p = subprocess.run([sys.executable, "-c", CHILD], env=dict(os.environ, MH_WALK_LINKS=v), capture_output=True,
                           text=True, timeout=600)
        assert p.returncode == 0, p.stdout + p.stderr
        got.append(p.stdout)
    assert got[0] == got[1]
