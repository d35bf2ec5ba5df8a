"""Duplicate removal on made-up hit lists against the oracle's sequential
walk, at the edges of the lanes per track (8) and of the blocks: track counts
around them, rows shorter and longer than the lanes, empty tracks, several
tracks sharing the same hits, a full row of the allocation-free entry."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _tracks(n, L, seed):
    """Families of up to five tracks that share some of their hits."""
    r = np.random.default_rng([seed, n, L])
    hits = np.full((n, L), -1, np.int32)
    n_found = r.integers(0 if n > 4 else 1, L + 1, size=n).astype(np.int32)
    n_hits = n * L + 1
    fresh = r.permutation(n_hits)[:n * L].reshape(n, L)
    family = r.integers(0, max(1, n // 3), size=n)
    pool = r.permutation(n_hits)[:(n // 3 + 1) * L].reshape(-1, L)
    for t in range(n):
        k = n_found[t]
        row = np.where(r.random(L) < r.uniform(0, 1), pool[family[t]], -1)
        used = set(row[row >= 0].tolist())
        for j in range(L):
            if row[j] < 0:
                row[j] = fresh[t, j] if fresh[t, j] not in used else -1
        row = row[row >= 0][:k]
        n_found[t] = row.size
        hits[t, :row.size] = row
    chi2 = r.uniform(1.0, 60.0, size=n).astype(np.float32)
    return hits, n_found, chi2, n_hits


@pytest.mark.parametrize("n,L", [(1, 1), (2, 32), (31, 7), (32, 8), (33, 9), (257, 17), (1025, 3), (3000, 31)])
def test_noalloc_lists_match_sequential_walk(n, L):
    import torch

    from paper_1906_11744_gb300 import _lib
    hits, n_found, chi2, n_hits = _tracks(n, L, 5)
    dev = torch.device("cuda:0")
    keep = torch.full((n,), 7, dtype=torch.uint8, device=dev)
    status = torch.full((1,), -9, dtype=torch.int32, device=dev)
    rc = _lib.kf_remove_duplicates_noalloc(n, L, n_hits, torch.from_numpy(hits).to(dev),
                                           torch.from_numpy(n_found).to(dev), torch.from_numpy(chi2).to(dev), 0.4,
                                           keep, status)
    assert rc == _lib.KF_OK
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle.dedup(hits, n_found, chi2.astype(np.float64), float(np.float32(0.4)))
    ref = np.where(n_found > 0, ref, 0)
    assert np.array_equal(keep.cpu().numpy(), ref)


def test_event_beyond_the_shared_memory_states():
    """An event of more tracks than the resolution holds in shared memory."""
    from kfhelp import tracker_for
    from synth import make_batch
    b = make_batch("c1b", tracks=25000)
    t = tracker_for(b)
    t.find_tracks()
    t.remove_duplicates()
    trk = t.get_tracks()
    t.close()
    assert b.n_seeds > 24576
    ref = oracle.dedup(trk["hits"], trk["n_found"], trk["chi2"].astype(np.float64), 0.5)
    assert np.array_equal(trk["keep"], ref)
    assert 0 < b.n_seeds - int(ref.sum()) < b.n_seeds
