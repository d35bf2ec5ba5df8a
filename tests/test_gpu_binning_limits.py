"""The largest grid of the grouped binning (12,288 buckets of one eta row per
event: 48 surfaces x 256 rows of 16,384 phi bins) and the smallest beyond it
(49 surfaces), which the general form takes.  Found tracks do not depend on the
grid; the per-event form is run too."""
import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_event", [0, 1])
@pytest.mark.parametrize("layers,surfaces", [(16, 48), (17, 49)])
def test_grid_at_the_bucket_limit(layers, surfaces, per_event):
    b = make_batch("c5", tracks=400, n_layers=layers, disk_z=tuple(125.0 + 8.0 * k for k in range(16)))
    assert b.det.n_surfaces == surfaces
    got = []
    for eta, phi in ((64, 1024), (256, 16384)):
        t = tracker_for(b, n_eta_bins=eta, n_phi_bins=phi, per_event=per_event)
        t.find_tracks()
        got.append(t.get_tracks())
        t.close()
    assert (got[0]["n_found"] > 3).any()
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k
