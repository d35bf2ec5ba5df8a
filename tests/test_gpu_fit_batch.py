"""A track's fit does not depend on how many others are fitted with it: up to
two listed tracks per SM the double-precision steps of the careful pass are
shared by a warp, above that each lane takes a track.  The same tracks alone,
with one more (the edge: 304 and 305 listed tracks on 152 SMs, every track of a
loose prior being listed) and among many have the same fit bit for bit: the two
forms do the same operations in the same order."""
import dataclasses

import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch
from synth.events import true_hit_lists
from test_gpu_careful import LOOSE_VAR

pytestmark = pytest.mark.gpu


def _make(kind):
    """(batch, hit lists, counts): seeds in an order in which any first part has listed tracks."""
    if kind == "disks":
        b = make_batch("c5")
    elif kind == "options":
        b = make_batch("c3", tracks=2500, field_cz=-3.0e-5, field_cr=-2.0e-5)
        x0 = np.random.default_rng(3).uniform(0.005, 0.06, size=(b.det.n_layers, 9)).astype(np.float32)
        b.det = dataclasses.replace(b.det, eloss=(7e-4,) * b.det.n_layers, x0_map=x0)
    elif kind == "loopers":
        b = make_batch("c3", tracks=60000)
    else:
        b = make_batch("c3", tracks=2500)
    lists, nh = true_hit_lists(b, 0, b.det.n_surfaces)
    sel = np.arange(b.n_seeds)
    if kind == "loopers":
        sel = np.argsort(-np.abs(b.params[3]))[:6000]
    else:
        for i in range(6):
            b.cov[i * 6 - i * (i - 1) // 2] = LOOSE_VAR[i]
    return b, sel, lists[b.seed_sim], nh[b.seed_sim]


def _fit(b, sel, lists, nh):
    from paper_1906_11744_gb300 import KF_FIT_GIVEN
    c = lambda a: np.ascontiguousarray(a[:, sel])  # noqa: E731
    s = dataclasses.replace(b, params=c(b.params), cov=c(b.cov), seed_hits=c(b.seed_hits), seed_sim=b.seed_sim[sel],
                            seed_off=np.array([0, len(sel)], np.int32))
    t = tracker_for(s)
    t.fit_tracks(KF_FIT_GIVEN, lists[sel], nh[sel])
    fit = t.get_fit()
    t.close()
    return fit


@pytest.mark.parametrize("kind", ["loose", "loopers", "options", "disks"])
def test_fit_independent_of_the_batch(kind):
    import torch
    b, sel, lists, nh = _make(kind)
    whole = _fit(b, sel, lists, nh)
    assert (whole["status"] == 0).mean() > 0.98
    edge = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    parts = [(0, n) for n in (1, 2, 150, edge, edge + 1)] + [(a, a + 300) for a in range(0, 1500, 300)]
    for a, e in parts:
        part = _fit(b, sel[a:e], lists, nh)
        for k in part:
            assert np.array_equal(part[k], np.asarray(whole[k])[..., a:e]), (a, e, k)
