"""Runs of empty reads: packing passes over them, wherever they lie, in about
the time that it takes without them, and finds the reads between them."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

E, R = 0, 1  # runs of empty reads, of reads of 150 bases


@pytest.mark.parametrize("runs", [
    [(E, 31), (R, 1), (E, 32), (R, 1), (E, 33), (R, 3), (E, 9000), (R, 1), (E, 64), (R, 1), (E, 255), (R, 40), (E, 256), (R, 1), (E, 257), (R, 2)],
    [(R, 5), (E, 1000), (R, 1), (E, 70_000)], [(E, 100_000)], [(E, 4097), (R, 27), (E, 8191), (R, 1), (E, 1), (R, 1), (E, 300)]],
    ids=["short", "at_the_end", "alone", "beside_tiles"])
def test_reads_between_empty_ones(runs):
    import torch

    import paper_1409_7208_gb300 as mh

    lens = np.concatenate([np.full(n, 150 * kind) for kind, n in runs])
    offs = np.concatenate([[0], np.cumsum(lens)])
    codes = np.random.default_rng(1).integers(0, 4, offs[-1])
    ascii = torch.from_numpy(np.frombuffer(b"ACGT", np.uint8)[codes].copy()).cuda()
    t = mh.mh_pack_reads(mh.Context(device=0), ascii, torch.from_numpy(offs).cuda()).tensors()
    full = np.flatnonzero(lens)
    assert t["n_frags"] == len(full) and t["n_packed"] == offs[-1]
    assert np.array_equal(t["frag_read"].cpu().numpy(), full)
    assert np.array_equal(t["frag_offs"].cpu().numpy(), np.append(offs[full], offs[-1]))
    padded = np.zeros(-(-len(codes) // 16) * 16, dtype=np.uint32)
    padded[:len(codes)] = codes
    want = (padded.reshape(-1, 16) << (30 - 2 * np.arange(16, dtype=np.uint32))).sum(axis=1, dtype=np.uint32)
    assert np.array_equal(t["packed"].cpu().numpy().view(np.uint32)[:len(want)], want)


@pytest.mark.parametrize("where", ["together", "mixed"])
def test_empty_reads_cost_little(where):
    import torch

    import paper_1409_7208_gb300 as mh

    ctx = mh.Context(device=0)
    reads, empty = 300_000, 3_000_000

    def best(lens):
        offs = np.concatenate([[0], np.cumsum(lens)])
        ascii = torch.full((int(offs[-1]),), ord("A"), dtype=torch.uint8, device="cuda")
        ascii[7] = ord("N")
        offs, times = torch.from_numpy(offs).cuda(), []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            r = mh.mh_pack_reads(ctx, ascii, offs)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
            r.free()
        return min(times)

    lens = np.zeros(reads + empty, dtype=np.int64)
    lens[(np.r_[:reads // 2, reads // 2 + empty:reads + empty]) if where == "together" else np.arange(reads) * 11] = 150
    # eleven times the reads: the offsets alone are more than half as much memory again
    assert best(lens) <= 3 * best(np.full(reads, 150))
