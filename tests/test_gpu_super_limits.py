"""Limits of counting by super-k-mers: the memory it takes where its bins do
not fit their tables (every bin left to the unit counting by MH_SUPER_HOT=0), and outputs whose
sizes were estimated too small (MH_SUPER_ESTIMATE: a share of the estimate,
and more bins left over in the first attempt than in the second).  Reads that
cover little sequence very deeply put many windows in few bins: sets that the
bins would mostly leave over go to the unit counting, the others do not."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code, args, env):
    p = subprocess.run([sys.executable, "-c", "import sys; sys.path.insert(0, %r)\n" % ROOT + code] + [str(a) for a in args],
                       env=dict(os.environ, **env), capture_output=True, text=True, timeout=900)
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout.split()


BUDGET = r"""
import hashlib
import synth, paper_1409_7208_gb300 as mh
k, reads, length, d = (int(x) for x in sys.argv[1:])
# little sequence: nearly every window is one of a few thousand
a, o = synth.uniform_genome_reads(k, 2000, reads, length, 0.0005)
n = reads * (length - k)
nw = 1 if k <= 31 else 2 if k <= 63 else 4
# the least budget that counts in memory: 24 nw + 12 bytes a window within 90 %
# of what the offsets of the fragments' windows leave of it
budget = int(n * 1.05 * (24 * nw + 12) / 0.9) + 8 * (reads + 1) + (1 << 20)
packed = mh.mh_pack_reads(mh.Context(device=0), a, o)
ctx = mh.Context(device=0, hbm_budget=budget, profile=True)
s = mh.mh_count_kmers(ctx, packed, k, d)
g, peak, prof = s.numpy(), ctx.memory()[1], ctx.profile()
assert peak <= budget and "bucket_hist" not in prof
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), "super_expand" in prof)
"""


@pytest.mark.parametrize("k", [31, 47, 99])
def test_all_bins_left_over_fit_the_in_memory_budget(k):
    old = _child(BUDGET, [k, 60_000, 150, 2], {"MH_SUPER": "0"})
    new = _child(BUDGET, [k, 60_000, 150, 2], {"MH_SUPER": "1", "MH_SUPER_HOT": "0"})
    assert new[0] == old[0] and (new[1], old[1]) == ("True", "False")


@pytest.mark.parametrize("k,windows,d", [(31, 2, 1), (31, 1, 2), (31, 2, 2), (47, 2, 2), (99, 2, 2)])
def test_a_record_a_window_or_two_fits_the_in_memory_budget(k, windows, d):
    args = [k, 6_000_000 // windows, k + windows, d]
    assert _child(BUDGET, args, {"MH_SUPER": "1"})[0] == _child(BUDGET, args, {"MH_SUPER": "0"})[0]


SAMPLED = r"""
import hashlib
import synth, paper_1409_7208_gb300 as mh
k, n_reads = int(sys.argv[1]), int(sys.argv[2])
a, o = synth.uniform_genome_reads(k, 3_000_000, n_reads, 150, 0.01)
ctx = mh.Context(device=0, profile=True)
s = mh.mh_count_kmers(ctx, mh.mh_pack_reads(ctx, a, o), k, 2)
g = s.numpy()
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), s.view().n_distinct, ctx.profile()["super_count"][0])
"""


@pytest.mark.parametrize("k,n_reads,probes", [(31, 300_000, 6), (31, 300_000, 128), (61, 400_000, 10), (61, 400_000, 128)])
def test_outputs_sized_too_small_are_made_again(k, n_reads, probes):
    # above 2^25 windows: the first bins counted, the others, the others again
    want = _child(SAMPLED, [k, n_reads], {})
    got = _child(SAMPLED, [k, n_reads], {"MH_SUPER_ESTIMATE": "1", "MH_SUPER_PROBES": str(probes)})
    assert got[:2] == want[:2] and (want[2], got[2]) == ("2", "3")


DEEP = r"""
import hashlib, time, torch
import synth, paper_1409_7208_gb300 as mh
genome, depth, k = (int(x) for x in sys.argv[1:])
a, o = synth.uniform_genome_reads(3, genome, genome * depth // 150, 150, 0.01)
ctx = mh.Context(device=0, profile=True)
reads = mh.mh_pack_reads(ctx, a, o)
s = mh.mh_count_kmers(ctx, reads, k, 2)
g, units = s.numpy(), "extract_canonical" in ctx.profile() or "extract_scatter" in ctx.profile()
ctx.set_profile(False)
times = []
for _ in range(6):
    s.free()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s = mh.mh_count_kmers(ctx, reads, k, 2)
    torch.cuda.synchronize()
    times.append(time.perf_counter() - t0)
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), g["n_distinct"], units, min(times))
"""


@pytest.mark.parametrize("genome,depth,k,units", [(30_000, 1000, 31, False), (100_000, 1000, 61, True), (300_000, 300, 47, False),
                                                  (30_000, 1000, 99, False), (3000, 5000, 61, False), (300_000, 30, 61, False)])
def test_deep_coverage_is_no_slower_than_the_unit_route(genome, depth, k, units):
    # a quarter more for what is done before the bins are given up
    new, old = (_child(DEEP, [genome, depth, k], e) for e in ({}, {"MH_SUPER": "0"}))
    assert new[:2] == old[:2] and (new[2], old[2]) == (str(units), "True")
    assert float(new[3]) <= 1.25 * float(old[3]), (new, old)


SORTS = r"""
import hashlib
import synth, paper_1409_7208_gb300 as mh
k = int(sys.argv[1])
a, o = synth.uniform_genome_reads(k, 1_500_000, 250_000, 150, 0.01)
ctx = mh.Context(device=0, profile=True)
s = mh.mh_count_kmers(ctx, mh.mh_pack_reads(ctx, a, o), k, 2)
g = s.numpy()
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), ctx.profile()["spread_fixup_kv"][0])
"""


@pytest.mark.parametrize("k", [31, 61, 99])
def test_pairs_of_left_over_bins_are_sorted_once(k):
    new, old = _child(SORTS, [k], {"MH_SUPER": "1", "MH_SUPER_HOT": "0"}), _child(SORTS, [k], {"MH_SUPER": "0"})
    assert new[0] == old[0] and (new[1], old[1]) == ("1", "1")


SATELLITE = r"""
import hashlib, time, torch
import numpy as np
import synth, paper_1409_7208_gb300 as mh
k = int(sys.argv[1])
# copies of one unit, a tenth of their bases changed: bins of very different sizes
rng = np.random.default_rng(2)
g = np.tile(rng.integers(0, 4, 171), 6000)
g = np.where(rng.random(len(g)) < 0.1, rng.integers(0, 4, len(g)), g)
at = rng.integers(0, len(g) - 150, 200_000)
b = g[at[:, None] + np.arange(150)]
b = np.where(rng.random(b.shape) < 0.01, rng.integers(0, 4, b.shape), b)
a = np.frombuffer(b"ACGT", np.uint8)[b].reshape(-1).copy()
ctx = mh.Context(device=0)
reads = mh.mh_pack_reads(ctx, a, np.arange(200_001, dtype=np.uint64) * 150)
times = []
for _ in range(6):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s = mh.mh_count_kmers(ctx, reads, k, 2)
    torch.cuda.synchronize()
    times.append(time.perf_counter() - t0)
g = s.numpy()
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), g["n_distinct"], min(times))
"""


@pytest.mark.parametrize("k", [31, 47, 61, 99])
def test_bins_of_very_different_sizes(k):
    new, old = _child(SATELLITE, [k], {}), _child(SATELLITE, [k], {"MH_SUPER": "0"})
    assert new[:2] == old[:2]
    assert float(new[2]) <= 1.25 * float(old[2]), (new, old)
