"""Loads and results at the edges of their forms: 127 events (offsets in the
launch's arguments) and 128 (offsets copied), and host arrays above the 16 MB
that the copy kernels take.  The same events alone, or the same arrays in
device memory, give the same results bit for bit."""
import dataclasses

import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("events", [127, 128])
def test_events_around_the_offsets_in_the_arguments(events, device):
    import torch
    dev = torch.device("cuda:0") if device else None
    b = make_batch("c1", n_events=events, tracks=31)
    t = tracker_for(b, device=dev)
    t.find_tracks()
    t.remove_duplicates()
    whole = t.get_tracks()
    t.close()
    for e in (0, 1, events // 2, events - 2, events - 1):
        s, h = slice(b.seed_off[e], b.seed_off[e + 1]), slice(b.hit_off[e], b.hit_off[e + 1])
        c = lambda a: np.ascontiguousarray(a[:, s])  # noqa: E731
        one = dataclasses.replace(b, x=b.x[h], y=b.y[h], z=b.z[h], layer=b.layer[h], params=c(b.params), cov=c(b.cov),
                                  seed_hits=c(b.seed_hits), hit_off=np.array([0, h.stop - h.start], np.int32),
                                  seed_off=np.array([0, s.stop - s.start], np.int32))
        t = tracker_for(one, device=dev)
        t.find_tracks()
        t.remove_duplicates()
        part = t.get_tracks()
        t.close()
        for k in part:
            whole_k = whole[k][s] if whole[k].shape[0] == b.n_seeds else whole[k][:, s]
            assert np.array_equal(part[k], whole_k), (e, k)


def test_host_arrays_above_the_copy_kernels_limit():
    import torch
    one, k = make_batch("c1", tracks=8000), 18
    rep = lambda a: np.concatenate([a] * k, axis=-1)  # noqa: E731
    b = dataclasses.replace(one, x=rep(one.x), y=rep(one.y), z=rep(one.z), layer=rep(one.layer), params=rep(one.params),
                            cov=rep(one.cov), seed_hits=rep(one.seed_hits),
                            hit_off=np.arange(k + 1, dtype=np.int32) * one.n_hits,
                            seed_off=np.arange(k + 1, dtype=np.int32) * one.n_seeds)
    assert min(16 * b.n_hits, 120 * b.n_seeds) > 16 << 20
    dev = torch.device("cuda:0")
    th, td = tracker_for(b), tracker_for(b, device=dev)
    th.find_tracks()
    td.find_tracks()
    host, device = th.get_tracks(), td.get_tracks(device=dev)
    assert sum(v.nbytes for v in host.values()) > 16 << 20
    for key in host:
        assert np.array_equal(host[key], device[key].cpu().numpy()), key
    th.close()
    td.close()
