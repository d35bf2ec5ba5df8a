"""Long careful lists: every track listed (a loose prior), or most of them with
double-precision steps (loopers), in batches of one event repeated, below and
above the size at which the adjoint's careful passes take wider blocks (128
tracks per SM) and beyond the largest grids (12 warps per SM, 32 tracks each).
The single event is checked against the oracle by tests/test_gpu_careful.py;
here every copy of it has the single event's fit bit for bit, and its gradient
norm-wise within the 1e-3 of the adjoint's parity test."""
import dataclasses

import numpy as np
import pytest

from kfhelp import tracker_for
from synth.events import true_hit_lists
from test_gpu_careful import _batch, _loopers

pytestmark = pytest.mark.gpu


def _repeat(b, k):
    rep = lambda a: np.concatenate([a] * k, axis=-1)  # noqa: E731
    return dataclasses.replace(b, x=rep(b.x), y=rep(b.y), z=rep(b.z), layer=rep(b.layer), params=rep(b.params),
                               cov=rep(b.cov), seed_hits=rep(b.seed_hits),
                               hit_off=np.arange(k + 1, dtype=np.int32) * b.n_hits,
                               seed_off=np.arange(k + 1, dtype=np.int32) * b.n_seeds)


def _run(b, lists, nh, stride):
    from paper_1906_11744_gb300 import KF_FIT_GIVEN
    t = tracker_for(b, ckpt_stride=stride)
    t.fit_tracks(KF_FIT_GIVEN, lists, nh)
    g_align = np.zeros((b.det.n_layers, 2), np.float32)
    g_hits = np.zeros((b.n_hits, 3), np.float32)
    g_seed = np.zeros((6, b.n_seeds), np.float32)
    t.fit_adjoint(g_align, g_hits, g_seed)
    fit = t.get_fit()
    t.close()
    return fit, g_align, g_hits, g_seed


@pytest.mark.parametrize("stride", [1, 4])
@pytest.mark.parametrize("kind,n,k", [("loose", 2500, 7), ("loose", 2500, 8), ("loose", 2500, 26),
                                      ("loopers", 1500, 12), ("loopers", 1500, 13)])
def test_repeated_event(kind, n, k, stride):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    one = _batch(n, True) if kind == "loose" else _loopers(n)
    if sms == 152:  # the sizes lie on both sides of the edges they are meant for
        assert (k * one.n_seeds < 128 * sms) == (k in (7, 12))
        assert k != 26 or k * one.n_seeds > 12 * 32 * sms
    lists, nh = true_hit_lists(one, 0, one.det.n_layers)
    lists, nh = lists[one.seed_sim], nh[one.seed_sim]
    f1, ga1, gh1, gs1 = _run(one, lists, nh, stride)
    f, ga, gh, gs = _run(_repeat(one, k), np.concatenate([lists] * k), np.concatenate([nh] * k), stride)
    for key in f1:
        a = np.asarray(f[key])
        for e in range(k):
            assert np.array_equal(a[..., e * one.n_seeds:(e + 1) * one.n_seeds], f1[key]), (key, e)
    scale = lambda r: 1e-3 * np.abs(r).max()  # noqa: E731
    assert np.abs(gh.reshape(k, -1, 3) - gh1).max() < scale(gh1)
    assert np.abs(gs.reshape(6, k, -1) - gs1[:, None]).max() < scale(gs1)
    assert np.abs(ga - k * ga1).max() < k * scale(ga1)
