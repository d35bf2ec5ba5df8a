"""The finding kernel's register budget where it is left to the library: above
the size at which it takes the capped kernel (600,000 candidate places), with
and without endcap disks, the results and the work counters are those of either
budget asked for."""
import numpy as np
import pytest

from kfhelp import tracker_for
from synth import make_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("config,events", [("c4", 8), ("c6", 8)])
def test_library_choice_above_its_threshold(config, events):
    b = make_batch(config, n_events=events)
    assert b.n_seeds * b.cfg["max_cands"] > 600000
    got = []
    for kw in (dict(), dict(block_threads=128), dict(block_threads=128, find_regcap=1)):
        t = tracker_for(b, **kw)
        t.find_tracks()
        got.append((t.get_tracks(), t.counters()))
        t.close()
    for trk, cnt in got[1:]:
        for k in trk:
            assert np.array_equal(trk[k], got[0][0][k]), k
        assert cnt == got[0][1]
