"""The finding kernel's register budget where it is left to the library: above
the size at which it takes the capped kernel (600,000 candidate places), with
and without endcap disks, the results and the work counters are those of either
budget asked for; and the two ways in which the careful pass takes on a seed."""
import dataclasses

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


def _low_pt(n, of, **kw):
    """The n seeds of lowest pT of an event: many of them meet a near-tangent crossing."""
    b = make_batch("c1", tracks=of, **kw)
    sel = np.sort(np.argsort(-np.abs(b.params[3]))[:n])
    c = lambda a: np.ascontiguousarray(a[:, sel])  # noqa: E731
    return dataclasses.replace(b, params=c(b.params), cov=c(b.cov), seed_hits=c(b.seed_hits), seed_sim=b.seed_sim[sel],
                               seed_off=np.array([0, n], np.int32))


@pytest.mark.parametrize("holes,cands", [(3, 6), (0, 10), (1, 16)])
@pytest.mark.parametrize("n,of,over", [(700, 9000, False), (1000, 60000, True)])
def test_given_up_seeds_with_and_without_records(n, of, over, holes, cands):
    """Seeds that the main pass gives up are taken on from its record (compiler's
    register count), searched again from the seed (capped kernel) or, beyond the
    records' room of n / 32 + 64, both: equal results and equal counters."""
    b = _low_pt(n, of)
    got = []
    for cap in (0, 1):
        t = tracker_for(b, max_cands=cands, max_holes=holes, block_threads=128, find_regcap=cap)
        t.find_tracks()
        got.append((t.get_tracks(), t.counters()))
        t.close()
    redone = got[0][1]["redone"]
    assert redone > n // 32 + 64 if over else 1 <= redone <= n // 32 + 64
    for k in got[0][0]:
        assert np.array_equal(got[0][0][k], got[1][0][k]), k
    assert got[0][1] == got[1][1]
