"""Which routes the radix sorts take, seen by their launches: a table of keys
crowded in their top bits is sorted by passes, not group by group."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CROWDED = r"""
import sys
sys.path.insert(0, %r)
import hashlib
import synth, paper_1409_7208_gb300 as mh
k, genome = int(sys.argv[1]), int(sys.argv[2])
# every substitution of a short sequence: keys that differ past their top bits only
a, o = synth.uniform_genome_reads(4, genome, 20_000, 150, 0.01)
ctx = mh.Context(device=0, profile=True)
reads = mh.mh_pack_reads(ctx, a, o)
ctx.profile_reset()
s = mh.mh_count_kmers(ctx, reads, k, 2)
g = s.numpy()
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), s.view().n, ctx.profile()["radix_onesweep"][0])
""" % ROOT


@pytest.mark.parametrize("k,genome", [(61, 300), (61, 1000), (61, 3000), (99, 300), (99, 1000)])
def test_crowded_small_wide_tables_take_few_launches(k, genome):
    def run(env):
        p = subprocess.run([sys.executable, "-c", CROWDED, str(k), str(genome)], env=dict(os.environ, **env),
                           capture_output=True, text=True, timeout=600)
        assert p.returncode == 0, p.stdout + p.stderr
        return p.stdout.split()
    got, full = run({}), run({"MH_SPREAD_KV_MIN": str(1 << 30)})
    assert got[:2] == full[:2] and 1 << 12 < int(got[1]) < 1 << 20
    # beside the full sort: the passes by the top bits, and two groups' sorts
    assert int(got[2]) <= 2.5 * int(full[2]) + 8, (got, full)
