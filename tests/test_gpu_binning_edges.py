"""Grids at the edges of the grouped binning: phi bins that are no multiple of
the four cells per store, one row per bucket, buckets just above the hits held
in registers, one-hit events.  Found tracks do not depend on the grid."""
import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch

pytestmark = pytest.mark.gpu


def _find(b, **cfg):
    t = tracker_for(b, **cfg)
    t.find_tracks()
    r = t.get_tracks()
    t.close()
    return r


@pytest.mark.parametrize("eta,phi,tracks", [(64, 1001, 700), (63, 1022, 700), (1, 1, 300), (5, 16384, 300),
                                            (200, 3, 300), (4, 2, 3300), (64, 1024, 1)])
def test_grid_shapes(eta, phi, tracks):
    b = make_batch("c1", tracks=tracks)
    ref = _find(b, n_eta_bins=64, n_phi_bins=20000)  # the general form
    got = _find(b, n_eta_bins=eta, n_phi_bins=phi)
    for k in ref:
        assert np.array_equal(ref[k], got[k]), k
