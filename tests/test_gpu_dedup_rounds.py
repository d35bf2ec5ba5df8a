"""The resolution rounds of duplicate removal at the edges of their shared
memory, on made-up hit lists against the oracle's sequential walk: more than
5,120 undecided tracks in an event whose states fit (the list's room), one more
and one fewer than that, and chains in which each decision waits for the one
before, in the shared list and beyond it."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _keep(hits, n_found, chi2, n_hits):
    import torch

    from paper_1906_11744_gb300 import _lib
    dev = torch.device("cuda:0")
    keep = torch.full((len(hits),), 7, dtype=torch.uint8, device=dev)
    status = torch.full((1,), -9, dtype=torch.int32, device=dev)
    tt = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    rc = _lib.kf_remove_duplicates_noalloc(len(hits), hits.shape[1], n_hits, tt(hits), tt(n_found), tt(chi2), 0.5,
                                           keep, status)
    assert rc == _lib.KF_OK
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return keep.cpu().numpy()


def _groups(n, undecided):
    """n tracks of 12 hits; `undecided` of them share eight with a better track of their group of three."""
    r = np.random.default_rng([n, undecided])
    lead = np.full(n, -1)
    lead[1:1 + 3 * (undecided // 2)].reshape(-1, 3)[:, 1:] = np.arange(1, 1 + 3 * (undecided // 2), 3)[:, None]
    if undecided % 2:
        lead[-1] = 0
    fresh = np.arange(n * 12, dtype=np.int32).reshape(n, 12)
    hits = fresh.copy()
    dup = lead >= 0
    hits[dup, :8] = hits[lead[dup], :8]
    used, inv = np.unique(hits, return_inverse=True)
    chi2 = r.uniform(1.0, 60.0, size=n).astype(np.float32)
    chi2[dup] += 100.0
    perm = r.permutation(n)
    return inv.reshape(n, 12).astype(np.int32)[perm], chi2[perm], used.size, int(dup.sum())


@pytest.mark.parametrize("n,undecided", [(15000, 5119), (15000, 5120), (15000, 5121), (16384, 10920)])
def test_undecided_tracks_around_the_lists_room(n, undecided):
    hits, chi2, n_hits, dup = _groups(n, undecided)
    assert dup == undecided and n_hits <= 262144
    n_found = np.full(n, 12, np.int32)
    ref = oracle.dedup(hits, n_found, chi2.astype(np.float64), 0.5)
    assert np.array_equal(_keep(hits, n_found, chi2, n_hits), ref)
    assert int(ref.sum()) == n - undecided


@pytest.mark.parametrize("n", [200, 5121, 5122, 16384])
def test_chain_of_decisions(n):
    """Track i shares six of ten hits with track i + 1: every other track is kept, each decided after the one before."""
    hits = (4 * np.arange(n)[:, None] + np.arange(10)).astype(np.int32)
    n_found = np.full(n, 10, np.int32)
    chi2 = np.linspace(1.0, 60.0, n).astype(np.float32)
    chi2 = np.maximum.accumulate(chi2)
    ref = oracle.dedup(hits, n_found, chi2.astype(np.float64), 0.5)
    got = _keep(hits, n_found, chi2, 4 * n + 10)
    assert np.array_equal(got, ref)
    assert np.array_equal(ref, (np.arange(n) + 1) % 2)
