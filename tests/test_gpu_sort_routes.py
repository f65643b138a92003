"""Which tiles and routes the radix sorts take, seen by their launches: with
MH_SORT_CHUNK_TILES=1 a scatter pass is a launch a tile.  The tile shapes of
one-word keys differ (16, 12 and 14 keys a thread), and small sorts keep their
own; a table of keys crowded in their top bits is sorted
by passes, not group by group.  And the tiles of large sorts on inputs small
enough for the oracle (MH_SORT_SMALL=0, MH_TINY_SORT=0), in chains of one and
three tiles: every key width, keys alone and pairs (with MH_SPREAD_KV_MIN=0 and
without)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHAPES = r"""
import sys
sys.path.insert(0, %r)
import synth, paper_1409_7208_gb300 as mh
k = int(sys.argv[1])
a, o = synth.uniform_genome_reads(9, int(sys.argv[2]), int(sys.argv[3]), 150, 0.01)
ctx = mh.Context(device=0, profile=True)
reads = mh.mh_pack_reads(ctx, a, o)
for shape in (-1, 0, 1, 2):
    mh.mh_set_count_plan(ctx, path=0, sort_shape=shape, unit_bits_delta=0, spread_bits_delta=0, bucket_bits=-1)
    ctx.profile_reset()
    mh.mh_count_kmers(ctx, reads, k, 2)
    print(ctx.profile()["radix_onesweep"][0])
""" % ROOT


def _launches(code, args, env):
    p = subprocess.run([sys.executable, "-c", code] + [str(x) for x in args], env=dict(os.environ, **env),
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr
    return [int(x) for x in p.stdout.split()]


def test_shapes_of_large_one_word_sorts_differ():
    # 2 million windows by the unit counting
    default, s0, s1, s2 = _launches(SHAPES, [31, 100_000, 17_000], {"MH_SUPER": "0", "MH_SORT_CHUNK_TILES": "1"})
    assert default == s0 < s2 < s1


@pytest.mark.parametrize("k", [31, 47, 99])
def test_the_default_shape_keeps_the_tiles_of_small_sorts(k):
    # 60 thousand windows and the pairs kept of them
    default, s0 = _launches(SHAPES, [k, 4000, 60_000 // (150 - k)], {"MH_SUPER": "0", "MH_SORT_CHUNK_TILES": "1"})[:2]
    assert default == s0


CROWDED = r"""
import sys
sys.path.insert(0, %r)
import hashlib, time, torch
import synth, paper_1409_7208_gb300 as mh
k, genome = int(sys.argv[1]), int(sys.argv[2])
# every substitution of a short sequence: keys that differ past their top bits only
a, o = synth.uniform_genome_reads(4, genome, 20_000, 150, 0.01)
ctx = mh.Context(device=0, profile=True)
reads = mh.mh_pack_reads(ctx, a, o)
ctx.profile_reset()
s = mh.mh_count_kmers(ctx, reads, k, 2)
g, launches = s.numpy(), ctx.profile()["radix_onesweep"][0]
ctx.set_profile(False)
times = []
for _ in range(8):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s = mh.mh_count_kmers(ctx, reads, k, 2)
    torch.cuda.synchronize()
    times.append(time.perf_counter() - t0)
print(hashlib.sha256(g["keys"].tobytes() + g["counts"].tobytes()).hexdigest(), s.view().n, launches, min(times))
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
    # and to find that out costs little
    assert float(got[3]) <= 1.25 * float(full[3]), (got, full)


@pytest.mark.parametrize("chunk", ["1", "3"])
@pytest.mark.parametrize("kv_min", ["0", str(1 << 30)])
def test_large_tiles_on_small_inputs_match_oracle(chunk, kv_min):
    from test_gpu_chunks import CHILD

    env = dict(os.environ, MH_SORT_SMALL="0", MH_TINY_SORT="0", MH_SORT_CHUNK_TILES=chunk, MH_SPREAD_KV_MIN=kv_min)
    p = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=900)
    assert p.returncode == 0 and "ok" in p.stdout, p.stdout + p.stderr


def test_small_and_large_tiles_differ():
    def run(env):
        return _launches(SHAPES, [47, 4000, 600], dict(env, MH_SUPER="0", MH_SORT_CHUNK_TILES="1"))[0]
    assert run({"MH_SORT_SMALL": "0"}) < run({})
